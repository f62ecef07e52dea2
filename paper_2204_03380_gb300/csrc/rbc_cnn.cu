// rbc_cnn.cu -- the learned random-boundary-noise denoiser: a 5-layer 3x3
// CNN (1 -> 32 -> 32 -> 32 -> 32 -> 1 channels, ReLU after layers 1-4, the
// input added to the last layer's output), bf16 operands with fp32
// accumulation.  Not in the paper: it stands in for stacking many random
// boundary realizations of an RTM image (Section 4.3's noise is incoherent
// between realizations).
//
// The 32-channel activations are bf16 and channel-group planar:
// [image][channel / 8][row][col][channel % 8] (16 bytes per pixel and group,
// so a row of one group is contiguous for the TMA copies and the tensor-core
// operands); one-channel images are [image][row][col].  Weights are stored
// [tap][out][in] (tap = 3 * dy + dx, dy, dx in 0..2 for offsets -1..1).
// The 32 -> 32 convolutions (three hidden layers, and their backward-data
// passes: the same kernel with the taps mirrored and the channel roles
// swapped, its epilogue applying the ReLU mask of the layer below) and the
// 32 -> 1 last layer run as implicit GEMMs on the 5th-generation tensor cores
// (tcgen05.mma, operands in shared memory, fp32 accumulators in tensor
// memory).  The one-channel first layer runs on the warp-level tensor cores
// (mma.sync m16n8k16, the 9 taps padded to K = 16): as its own kernel in the
// training forward (its output is kept for the backward pass), inside the
// second layer's kernel for inference.  The weight gradients of
// the 32 -> 32 layers run on tcgen05 too (four rows of one operand against two
// of the other per MMA); those of the one-channel end layers on mma.sync with the taps
// on M.  Persistent blocks add their sums to the fp32 gradient once each.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <cstdlib>
#include <cstring>

#include "../../include/rbc.h"
#include "rbc_internal.cuh"

using rbc::griddep_launch;
using rbc::griddep_wait;
using rbc::launch_pdl;

namespace rbc {
int set_error(int code, const char *msg);  // rbc_abi.cu
void add_launches(long long n);
}

namespace {

constexpr int C = 32;           // hidden channels
// parameter offsets (fp32 master copy): W1 b1 W2 b2 W3 b3 W4 b4 W5 b5
constexpr int kW1 = 0, kB1 = kW1 + 9 * C, kW2 = kB1 + C, kB2 = kW2 + 9 * C * C, kW3 = kB2 + C,
              kB3 = kW3 + 9 * C * C, kW4 = kB3 + C, kB4 = kW4 + 9 * C * C, kW5 = kB4 + C, kB5 = kW5 + 9 * C,
              kNParams = kB5 + 1;

__device__ __forceinline__ void mma16816(float *c, const uint32_t *a, const uint32_t *b) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

enum { kHidden = 0, kLast = 1, kBackData = 2, kFused = 3 };

// The one-channel first layer (1 -> 32 channels, and the last layer's
// backward-data pass) on the warp-level tensor cores:
//   wt [tap][32] (bf16);  MODE kHidden: relu(conv + bias);  kBackData: conv where the sign bits are set
// Per 16 pixels of a row, one m16n8k16 MMA per group of 8 output channels with K = the 9 taps
// (padded to 16, zero weights): the im2col operand A[pixel][tap] is gathered
// from the staged halo straight into the A fragments, the weights are the B
// fragments, held in registers for the whole kernel (the bias is the
// accumulator's initial value).  A block of 8 warps covers 8 rows x 128
// pixels (one warp per row); persistent blocks prefetch the next tile's halo
// into registers.  The output fragment of lane (g, t) holds channels
// 8n + 2t, 8n + 2t + 1 of pixels g and g + 8: 4-byte pieces of the pixels'
// 16-byte channel groups, stored 128 contiguous bytes per warp and group
// (rounded and clamped at zero by one conversion for the forward layer;
// masked by the layer's sign bits for the backward-data pass).
//
// Sign bits: for every pixel of a layer's output 32 bits of which channels are
// positive, written beside it in the training forward and read by the backward-data pass in place of
// the activation (4 bytes per pixel, not 64).  Bit i is channel 2 i, bit 16 + i channel
// 2 i + 1: a packed comparison of two channels contributes both by one mask.
// The backward-data kernels of 8 x 512^2 took 39 us (this one) and 80 us (32 -> 32)
// reading the activation, 23 and 44 with the bits; writing them costs the forward
// layers nothing that was measured.
// Tile counts are ints: a tile holds 1024 pixels of 64-byte activations.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

constexpr int kM1R = 8, kM1C = 128;               // tile rows, columns
constexpr int kM1HW = kM1C + 2, kM1HP = (kM1R + 2) * kM1HW;  // halo columns, halo values
// halo row pitch in shared memory (2-byte values): 72 words, 8 banks apart,
// so the A-fragment gathers of a warp (three halo rows) are conflict-free
constexpr int kM1P = 144;
constexpr int kM1Pre = (kM1HP + 255) / 256;       // halo values per thread
__device__ __forceinline__ uint32_t pack_u16(uint16_t lo, uint16_t hi) { return (uint32_t)lo | ((uint32_t)hi << 16); }
// {lo, hi} rounded to bf16 (and clamped at zero for kRelu) in one 4-byte word
template <bool kRelu>
__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
  uint32_t r;
  if (kRelu) asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// 0xffff where a half of the pair is positive
__device__ __forceinline__ uint32_t positive(uint32_t pair) {
  return __hgt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&pair), __float2bfloat162_rn(0.f));
}
// 0xffff for the set ones of sign bits i and 16 + i (i a constant)
__device__ __forceinline__ uint32_t spread(uint32_t bits, int i) {
  const uint32_t t = bits << (i < 8 ? 7 - i : 15 - i);  // to the top of bytes 0 and 2, or 1 and 3
  uint32_t r;  // selectors 8 + k replicate byte k's top bit
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(t), "r"(i < 8 ? 0xaa88u : 0xbb99u));
  return r;
}

template <int MODE>
__global__ void __launch_bounds__(256, 3) k_conv_1to32(const float *__restrict__ in, __nv_bfloat16 *__restrict__ in16,
                                                        const __nv_bfloat16 *__restrict__ wt,
                                                        const float *__restrict__ bias,
                                                        uint32_t *__restrict__ bits,
                                                        __nv_bfloat16 *__restrict__ out, int nimg, int H, int W) {
  __shared__ __align__(16) uint16_t s_x[2][(kM1R + 2) * kM1P];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int ntx = (W + kM1C - 1) / kM1C, tpi = ntx * ((H + kM1R - 1) / kM1R), ntiles = tpi * nimg;
  const long long HWp = (long long)H * W;
  const uint16_t *win = reinterpret_cast<const uint16_t *>(wt);
  griddep_wait();
  griddep_launch();
  // B fragments: B[k][co] = w[tap k][co] for k < 9, zero above
  uint32_t bf[4][2];
  float2 bs[4];
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const int co = 8 * n + g;
    bf[n][0] = pack_u16(win[(2 * t) * 32 + co], win[(2 * t + 1) * 32 + co]);
    bf[n][1] = t == 0 ? pack_u16(win[8 * 32 + co], 0) : 0u;
    bs[n] = MODE == kHidden ? make_float2(bias[8 * n + 2 * t], bias[8 * n + 2 * t + 1]) : make_float2(0.f, 0.f);
  }
  // halo offsets of this lane's taps: 2t, 2t + 1 (and 8 for t = 0), tap = 3 dy + dx
  const int o0 = ((2 * t) / 3) * kM1P + (2 * t) % 3, o1 = ((2 * t + 1) / 3) * kM1P + (2 * t + 1) % 3;
  constexpr int o8 = 2 * kM1P + 2;
  auto origin = [&](int tt, int &img, int &y0, int &x0) {
    img = tt / tpi;
    const int rem = tt - img * tpi, ty = rem / ntx;
    y0 = ty * kM1R;
    x0 = (rem - ty * ntx) * kM1C;
  };
  auto fetch = [&](int img, int y0, int x0, float *v) {
    const float *src = in + (long long)img * HWp;
#pragma unroll
    for (int k = 0; k < kM1Pre; ++k) {
      const int i = tid + 256 * k, r = i / kM1HW;
      const int yy = y0 + r - 1, xx = x0 + (i - r * kM1HW) - 1;
      v[k] = (i < kM1HP && (unsigned)yy < (unsigned)H && (unsigned)xx < (unsigned)W) ? src[(long long)yy * W + xx]
                                                                                      : 0.f;
    }
  };
  // rounded to bf16; the forward layer also writes the tile's own pixels to in16
  auto park = [&](const float *v, int b, int img, int y0, int x0) {
#pragma unroll
    for (int k = 0; k < kM1Pre; ++k) {
      const int i = tid + 256 * k, r = i / kM1HW, c = i - r * kM1HW;
      if (i < kM1HP) {
        const __nv_bfloat16 h = __float2bfloat16(v[k]);
        s_x[b][r * kM1P + c] = __bfloat16_as_ushort(h);
        if (MODE == kHidden && r >= 1 && r <= kM1R && c >= 1 && c <= kM1C && y0 + r - 1 < H && x0 + c - 1 < W)
          in16[img * HWp + (long long)(y0 + r - 1) * W + x0 + c - 1] = h;
      }
    }
  };
  // kBackData: sign bits of this warp's row, pixels lane, lane + 32, ..
  auto fetch_bits = [&](int img, int y0, int x0, uint32_t *m) {
    if constexpr (MODE == kBackData) {
#pragma unroll
      for (int k = 0; k < kM1C / 32; ++k) {
        const int xx = x0 + lane + 32 * k;
        m[k] = (y0 + warp < H && xx < W) ? bits[img * HWp + (long long)(y0 + warp) * W + xx] : 0u;
      }
    }
  };
  float v[kM1Pre];
  uint32_t sb[kM1C / 32] = {}, sb_n[kM1C / 32] = {};
  int img = 0, y0 = 0, x0 = 0;
  if ((int)blockIdx.x < ntiles) {
    origin(blockIdx.x, img, y0, x0);
    fetch(img, y0, x0, v);
    fetch_bits(img, y0, x0, sb);
    park(v, 0, img, y0, x0);
  }
  uint32_t *o32 = reinterpret_cast<uint32_t *>(out);
  int b = 0;
  for (int tt = blockIdx.x; tt < ntiles; tt += gridDim.x, b ^= 1) {
    const int tn = tt + gridDim.x;
    int img_n = 0, y0_n = 0, x0_n = 0;
    if (tn < ntiles) {  // in flight during this tile
      origin(tn, img_n, y0_n, x0_n);
      fetch(img_n, y0_n, x0_n, v);
      fetch_bits(img_n, y0_n, x0_n, sb_n);
    }
    const int y = y0 + warp;
    const int nx = min(kM1C, W - x0);  // columns of the tile inside the image
    __syncthreads();  // s_x[b] holds tile tt
    if (y < H) {
      const uint16_t *sr = s_x[b] + warp * kM1P + g;
      // 4-byte piece t of pixel (y, x0 + g) in each channel group
      uint32_t *orow[4];
#pragma unroll
      for (int n = 0; n < 4; ++n) orow[n] = o32 + (((long long)img * 4 + n) * HWp + (long long)y * W + x0 + g) * 4 + t;
#pragma unroll
      for (int sg = 0; sg < kM1C / 16; ++sg) {
        if (16 * sg >= nx) break;
        const uint16_t *p0 = sr + 16 * sg, *p1 = p0 + 8;
        uint32_t a[4];
        a[0] = pack_u16(p0[o0], p0[o1]);
        a[1] = pack_u16(p1[o0], p1[o1]);
        a[2] = t == 0 ? (uint32_t)p0[o8] : 0u;
        a[3] = t == 0 ? (uint32_t)p1[o8] : 0u;
        float d[4][4];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          d[n][0] = d[n][2] = bs[n].x;
          d[n][1] = d[n][3] = bs[n].y;
          mma16816(d[n], a, bf[n]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // pixels g (h = 0) and g + 8
          const int px = 16 * sg + 8 * h;
          const bool in = px + g < nx;
          uint32_t w = 0;  // this pixel's sign bits (kBackData: moved down by t)
          if (MODE == kBackData) w = __shfl_sync(0xffffffffu, sb[sg >> 1], (16 * (sg & 1) + 8 * h) | g) >> t;
#pragma unroll
          for (int n = 0; n < 4; ++n) {
            uint32_t r;
            if (MODE == kHidden) {
              r = cvt_bf16x2<true>(d[n][2 * h], d[n][2 * h + 1]);
              w |= positive(r) & (0x00010001u << (4 * n));
            } else {
              r = cvt_bf16x2<false>(d[n][2 * h], d[n][2 * h + 1]) & spread(w, 4 * n);
            }
            if (in) orow[n][px * 4] = r;
          }
          if (MODE == kHidden) {
            w <<= t;
            w |= __shfl_xor_sync(0xffffffffu, w, 1);
            w |= __shfl_xor_sync(0xffffffffu, w, 2);
            if (in && t == 0) bits[img * HWp + (long long)y * W + x0 + px + g] = w;
          }
        }
      }
    }
    if (tn < ntiles) {  // read two tiles on, after the next barrier
      park(v, b ^ 1, img_n, y0_n, x0_n);
#pragma unroll
      for (int k = 0; k < kM1C / 32; ++k) sb[k] = sb_n[k];
      img = img_n;
      y0 = y0_n;
      x0 = x0_n;
    }
  }
}

// ---------------------------------------------------------------------------
// 32 -> 32 channel layers on the 5th-generation tensor cores (tcgen05).
//
// A tile is R output rows x 126 columns of one image.  The accumulator
// of output row rr is a 128 (pixels) x 32 (channels) fp32 matrix in tensor
// memory:
//   D_rr[px][co] = sum_(dy, dx) sum_ci halo[rr + dy][px + dx][ci] * w[dy][dx][co][ci].
// Halo row h enters the accumulators of up to three output rows (rr = h - dy,
// dy = 0, 1, 2), each time with the same shifted operand and a different
// weight slice.  So the MMAs run per (halo row h, dx, half of the input
// channels) with M = 128 pixels, K = 16 channels and N = 32 x (number of
// output rows h reaches): B stacks the weights of those dy values, and the
// output rows' accumulators sit in tensor memory in descending row order
// (row rr at column (R - 1 - rr) * 32), so the N columns of one MMA are
// exactly the accumulators it feeds.  Against one N = 32 MMA per (row, tap,
// half) this reads each shifted halo operand once instead of up to three
// times: 6 (R + 2) MMAs per tile instead of 18 R, and 40 % less
// shared-memory operand traffic at R = 4.  Every MMA accumulates; the
// epilogue clears each accumulator after reading it.
// Both operands sit in shared memory in the no-swizzle K-major layout: a
// "core matrix" is 8 rows of 16 bytes (8 channels) stored contiguously.  The
// activations are kept channel-group planar in memory ([image][group of 8
// channels][row][column][8]), so one 4-D TMA copy (rows of 8-byte elements)
// lands a tile's halo as four planes (one per channel group) of halo pixels
// in row-major order at 16 bytes each: 8 consecutive pixels of any halo row
// are one core matrix, and
// the operand of a shifted tap is the same planes with the start address
// moved by (h * 128 + dx) * 16 bytes (stride between 8-pixel groups 128
// bytes, between channel groups one plane).  Weights in shared memory:
// [dx][ci / 8][dy][co][8], so the 96 (dy, co) rows of one (dx, ci group) are
// consecutive core matrices (stride 128 bytes) and the two channel groups of a
// K = 16 slice are 1536 bytes apart.
//
// Per block (one per SM, persistent over tiles), three roles: warp kTcEpi
// streams each tile's halo (zero-filled outside the image) into a shared-
// memory ring of tc_units(R) half tiles (in the fused first-layer mode, builder
// warps compute it there instead); the next warp issues the 6 (R + 2)
// MMAs of a tile into one of two tensor-memory accumulators and commits them
// to the ring's "empty" and the accumulator's "full" barrier; warps 0 ..
// kTcEpi - 1 (two per tensor-memory lane quarter, one pixel per thread, half
// of the rows each) drain the other accumulator with tcgen05.ld, apply the
// epilogue (the backward-data pass reads the sign bits of the layer below a
// tile ahead) and store.  Copies of the next tiles,
// MMAs of tile k and the epilogue of tile k-1 overlap.  Every wait is bounded; a
// block that gives up flags the error word and stops.
// A tile is kTcOut = 126 output columns: its halo row is then 128 pixels of
// 16 bytes, 2 KB, which one tensor copy moves as 256 8-byte elements (the
// box limit), against a box whose innermost dimension is one pixel's 16
// bytes; measured on GB300 streaming such halos on every SM: 9.2 TB/s for
// the 2 KB rows, 4.4 TB/s for the 16-byte rows.  The MMAs keep M = 128:
// rows 126 and 127 of a shifted operand run into the next halo row and
// their outputs are discarded.
constexpr int kTcOut = 126;                                  // output columns per tile
constexpr int kTcHW = 128;                                   // halo row width (pixels)
constexpr int kTcWBytes = 9 * 4 * 32 * 16;                   // weights, 18432 B
constexpr long long kTcWaitCycles = 4000000000LL;            // about two seconds
constexpr int kTcEpi = 8;                                    // epilogue warps
// Tiles of R output rows: R = 8 fills tensor memory with the two accumulator buffers.
// Measured with a ring of whole tiles at 32 x 512^2 with 126-column tiles (inference / training step):
// R = 8 0.951 / 5.20 ms, R = 6 0.969 / 5.37 ms, R = 4 1.071 / 5.49 ms; with
// 128-column tiles and the 16-byte-row halo copy: R = 6 1.14 / 5.51 ms, R = 4
// 1.18 / 5.57 ms, R = 4 with 4 epilogue warps 1.23 / 5.88 ms.
constexpr int kTcR = 8, kTcRs = 4;  // rows per tile; of small images (tile_rows)
// The ring holds units of half a tile's halo (four planes of tc_ur(R) rows of
// 128 pixels), so that a copy starts when half a tile's MMAs are done.  Three units
// of five rows: more in flight only crowds L2 when the layer's data do not fit
// there.  Inference of 8 x 512^2 / 32 x 512^2 / 64 x 400 x 800, us: three units 192 /
// 681 / 1511, four 190 / 697 / 1602, five 193 / 716 / 1629; two whole tiles 203 / 714 /
// 1559; seven two-row units 187 / 675 / 1579.
constexpr int kTcTU = 2;  // units per tile
constexpr int tc_ur(int R) { return (R + 2) / kTcTU; }
constexpr int tc_plane(int R) { return tc_ur(R) * kTcHW * 16; }
constexpr int tc_units(int R) { return R <= 4 ? 6 : 3; }
constexpr int kTcTail = 512;  // bias, barriers, flags
constexpr int tc_smem(int R) { return kTcWBytes + tc_units(R) * 4 * tc_plane(R) + kTcTail; }
static_assert((kTcR + 2) % kTcTU == 0 && (kTcRs + 2) % kTcTU == 0, "a tile is whole units");
static_assert(2 * 8 * 32 <= 512, "two accumulator buffers must fit in tensor memory");
static_assert(128 + 8 * (2 * tc_units(kTcRs) + 4) + 8 <= kTcTail, "bias and barriers fit behind the ring");

// One lane of the warp, by elect.sync, in a warp chosen by a uniform test: the
// compiler then has what an MMA's issue needs in uniform registers.  A thread
// chosen by its lane number issued one MMA in 70 - 76 cycles where the
// operands' reads take 42 - 52 (hidden layer of 8 x 512^2 54 -> 52 us, last layer
// 45 -> 34; with the ring below 42 and 31).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  // no swizzle; start, leading (K) and stride (M/N) byte offsets in 16-byte
  // units; bits 46-47 = 1 (descriptor version of this architecture)
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// kind::f16 instruction descriptor: fp32 accumulator, bf16 A and B, both
// K-major, M = 128, N = n (a multiple of 16, at most 256).
constexpr uint32_t tc_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}


__device__ __forceinline__ void tmem_ld32(uint32_t ta, float *v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(ta));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 32; ++c) v[c] = __uint_as_float(r[c]);
}

// Clear 32 columns of this warp's 32 tensor-memory lanes (completion by
// tcgen05.wait::st).
__device__ __forceinline__ void tmem_zero32(uint32_t ta) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,"
      "%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(ta), "r"(0u)
      : "memory");
}

__device__ __forceinline__ void tc_mbar_init(uint32_t b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(count) : "memory");
}
__device__ __forceinline__ void tc_arrive(uint32_t b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(b) : "memory");
}
__device__ __forceinline__ bool tc_try(uint32_t b, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(b), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait that gives up when another role of the block has flagged an
// abort, and flags one itself when its time runs out.
__device__ __forceinline__ bool tc_wait(uint32_t b, uint32_t parity, volatile int *abort_blk) {
  if (tc_try(b, parity)) return true;
  const long long t0 = clock64();
  while (!tc_try(b, parity)) {
    if (*abort_blk) return false;
    if (clock64() - t0 > kTcWaitCycles) {
      *abort_blk = 1;
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void tc_tma4(uint32_t dst, const CUtensorMap *tm, int c0, int c1, int c3, uint32_t bar) {
  // coordinates (8-byte element along the row, y, group 0, image)
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(0), "r"(c3), "r"(bar)
      : "memory");
}

// Tensor-memory columns to allocate for c columns (a power of two >= 32).
constexpr int tmem_cols(int c) { return c <= 32 ? 32 : c <= 64 ? 64 : c <= 128 ? 128 : c <= 256 ? 256 : 512; }

__device__ __forceinline__ float tmem_ld1(uint32_t ta) {
  uint32_t r;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(ta));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  return __uint_as_float(r);
}
__device__ __forceinline__ void tmem_zero1(uint32_t ta) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(ta), "r"(0u) : "memory");
}

// Store four 8 x 8 bf16 matrices in the fragment layout of an MMA's result; lane 8 j + r gives the address of
// row r of matrix j.
__device__ __forceinline__ void stm_x4(uint32_t sa, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(sa), "r"(r0), "r"(r1), "r"(r2),
               "r"(r3)
               : "memory");
}

//   MODE kHidden:   out = relu(conv(in) + bias)                        (32 -> 32)
//   MODE kBackData: out = conv(in) where the sign bits are set   (weights mirrored and transposed)
//   MODE kLast:     out_f = resid + conv(in) + bias                    (32 -> 1)
//   MODE kFused:    out = relu(conv(a1) + bias) with a1 = relu(conv1(x1) + b1)
//                   computed in the block (the first two layers, for inference)
// The last layer's single output channel is padded to N = 16 per output row
// (the smallest N of an M = 128 MMA); the 15 padding channels have zero
// weights, so their accumulators stay zero and only channel 0 is read out.
// kTcEpi epilogue warps: warp e drains TMEM lane quarter e % 4 (pixels
// 32 (e % 4) .. +31) for the output rows of its share (R * 4 / kTcEpi rows,
// starting at row (e / 4) * R * 4 / kTcEpi); warps kTcEpi .. kTcEpi +
// tc_nprod(MODE, R) - 1 are the producers, the next warp the MMA issuer.
//
// kFused: instead of the tensor copy of a stored first-layer output, R + 2
// builder warps compute it over the tile's halo (R + 2 rows x 128 pixels,
// one row per warp) into the ring stage, in the layout the copy would have
// produced: the fp32 one-channel input's halo (R + 4 rows x 130 pixels,
// prefetched a tile ahead into registers, rounded to bf16) is parked in
// shared memory, and each 16 pixels of a halo row are one m16n8k16 MMA per 8
// channels as in k_conv_1to32 (taps padded to K = 16, bias as the
// accumulator's start, relu and rounding in one conversion), stored by
// stmatrix as rows of 16 bytes (a pixel's channel group); 64 pixels' operands are
// gathered ahead, and two parked halos leave one barrier per tile.  Outside
// the image the stage holds zeros (the second
// layer's padding).  These warps bound the fused layers: mma.sync and tcgen05
// take turns on the tensor pipe (32 x 512^2: 235 us; 175 without the mma.sync).  The builders then make their writes visible to the
// tensor cores and arrive on the stage's "full" barrier.  The first layer's
// output never passes through global memory.
constexpr int tc_nprod(int mode, int R) { return mode == kFused ? R + 2 : 1; }
constexpr int tc_threads(int mode, int R) { return 32 * (kTcEpi + tc_nprod(mode, R) + 1); }
constexpr int kFxR = 4;                  // x halo rows beyond the tile's R (two on each side)
constexpr int kFxC = kTcHW + 2;          // x halo columns (x0 - 2 .. x0 + 127)
constexpr int kFxP = 144;                // x halo row pitch (2-byte values; conflict-free gathers)
constexpr int tc_fx_bytes(int R) { return (R + kFxR) * kFxP * 2; }
constexpr int tc_fx_vals(int R) { return (R + kFxR) * kFxC; }  // x halo values of a tile
constexpr int tc_smem_mode(int mode, int R) { return tc_smem(R) + (mode == kFused ? 2 * tc_fx_bytes(R) : 0); }
static_assert(tc_smem_mode(kFused, kTcR) <= 227 * 1024, "the fused ring must fit in shared memory");

// Strides (in values) of the one-channel images: from image to image and from
// row to row, of the input and of the output.
struct Img {
  long long xi, xr, yi, yr;
};

template <int MODE, int R>
__global__ void __launch_bounds__(tc_threads(MODE, R), 1) k_conv_tc(const __grid_constant__ CUtensorMap tm_in,
                                                    const void *__restrict__ wt_,
                                                    const float *__restrict__ bias,
                                                    uint32_t *__restrict__ bits,
                                                    __nv_bfloat16 *__restrict__ out, float *out_f,
                                                    const float *xin, const Img st, int nimg, int H, int W,
                                                    int rev, int *err, const float *__restrict__ w1 = nullptr,
                                                    const float *__restrict__ b1 = nullptr) {
  constexpr bool kHid = MODE == kHidden || MODE == kFused;  // relu(conv + bias) epilogue
  constexpr int kMma = kTcEpi + tc_nprod(MODE, R);             // the MMA issuer warp
  constexpr int NCO = MODE == kLast ? 16 : 32;  // output channels per row accumulator
  constexpr int WCG = 3 * NCO * 16;              // weight bytes per (dx, channel group)
  constexpr int WDX = 4 * WCG;                   // weight bytes per dx
  constexpr int BUF = R * NCO;             // accumulator columns per tile buffer
  constexpr int TCOLS = tmem_cols(2 * BUF);
  constexpr int PLANE = tc_plane(R), NU = tc_units(R), TU = kTcTU, UR = tc_ur(R), UNIT = 4 * PLANE;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s_w = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t s_h = s_w + kTcWBytes;  // halo ring
  unsigned char *tail = smem + kTcWBytes + NU * UNIT;
  float *s_bias = reinterpret_cast<float *>(tail);
  // barriers: full[NU], empty[NU], tfull[2], tempty[2]
  uint64_t *bars = reinterpret_cast<uint64_t *>(tail + 128);
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * NU + 4);
  volatile int *abort_blk = reinterpret_cast<volatile int *>(tslot + 1);
  const uint32_t b0 = (uint32_t)__cvta_generic_to_shared(bars);
  auto full = [&](int i) { return b0 + 8u * i; };
  auto empty = [&](int i) { return b0 + 8u * (NU + i); };
  auto tfull = [&](int i) { return b0 + 8u * (2 * NU + i); };
  auto tempty = [&](int i) { return b0 + 8u * (2 * NU + 2 + i); };
  // The prologue (weights, barriers, tensor memory: about 3 us) overlaps the
  // previous layer's launch: an image of 200 x 200 took 43 us, 30 with it.
  // Only the weights are read in it: whatever wrote them comes before the first layer,
  // which the layers before this one have waited for (the fused first layers wait here).
  if (MODE == kFused) griddep_wait();
  // weights [tap][co][ci] (tap = 3 dy + dx) -> [dx][ci / 8][dy][co][8]; the forward
  // layers round the fp32 parameters here (a launch of its own for that cost a small
  // image 4 us), the backward-data pass copies its mirrored bf16 weights
  if (MODE == kLast) {
    for (int i = tid; i < 9 * 4 * (NCO - 1); i += blockDim.x) {  // padding channels 1..15: zero
      const int co = 1 + i % (NCO - 1), r = i / (NCO - 1), j = r & 3, t = r >> 2;
      *reinterpret_cast<uint4 *>(smem + (t % 3) * WDX + j * WCG + (t / 3) * NCO * 16 + co * 16) =
          make_uint4(0u, 0u, 0u, 0u);
    }
    const float *wt = static_cast<const float *>(wt_);
    for (int i = tid; i < 9 * 32; i += blockDim.x) {
      const int ci = i & 31, t = i >> 5;
      *reinterpret_cast<__nv_bfloat16 *>(smem + (t % 3) * WDX + (ci >> 3) * WCG + (t / 3) * NCO * 16 + (ci & 7) * 2) =
          __float2bfloat16(wt[i]);
    }
  } else if (MODE == kBackData) {
    const __nv_bfloat16 *wt = static_cast<const __nv_bfloat16 *>(wt_);
    for (int i = tid; i < 9 * 32 * 4; i += blockDim.x) {
      const int j = i & 3, co = (i >> 2) & 31, t = i >> 7, dy = t / 3, dx = t % 3;
      cp_async16(s_w + dx * WDX + j * WCG + dy * NCO * 16 + co * 16, wt + (t * 32 + co) * 32 + j * 8, true);
    }
  } else {
    const float *wt = static_cast<const float *>(wt_);
#pragma unroll 8
    for (int i = tid; i < 9 * 32 * 32; i += tc_threads(MODE, R)) {
      const int ci = i & 31, co = (i >> 5) & 31, t = i >> 10, dy = t / 3, dx = t % 3;
      *reinterpret_cast<__nv_bfloat16 *>(smem + dx * WDX + (ci >> 3) * WCG + dy * NCO * 16 + co * 16 + (ci & 7) * 2) =
          __float2bfloat16(wt[i]);
    }
  }
  if (kHid && tid < 32) s_bias[tid] = bias[tid];
  if (MODE == kLast && tid == 0) s_bias[0] = bias[0];
  if (tid == 0) {
    *abort_blk = 0;
    for (int i = 0; i < NU; ++i) {
      tc_mbar_init(full(i), MODE == kFused ? 32 * UR : 1);
      tc_mbar_init(empty(i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc_mbar_init(tfull(i), 1);
      tc_mbar_init(tempty(i), 32 * kTcEpi);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
        (uint32_t)__cvta_generic_to_shared(tslot)), "r"(TCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);  // (uniform: see elect_one)
  if (warp < 4) {  // every MMA accumulates: both accumulator buffers start at zero
#pragma unroll 1
    for (int c = 0; c < 2 * BUF; c += 32) tmem_zero32(tmem + ((uint32_t)(warp * 32) << 16) + c);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (MODE != kFused) griddep_wait();
  griddep_launch();
  // (32-bit tile numbers: a tile holds at least one pixel of some 400 bytes of workspace)
  const int ntx = (W + kTcOut - 1) / kTcOut, tpi = ntx * ((H + R - 1) / R), ntiles = tpi * nimg;
  // Persistent blocks over the tiles, x fastest (a contiguous y-fastest range per block lost: 1.36
  // against 1.27 ms per 32 x 512^2 inference).  rev: from the last tile to the
  // first.  Consecutive layers run in opposite directions, so that a layer begins with what the one
  // before wrote last and L2 still holds: 8 x 512^2 inference 210 -> 203 us,
  // training step 808 -> 786.
  auto tile_xy = [&](int t, int &img, int &y0, int &x0) {
    if (rev) t = ntiles - 1 - t;
    img = t / tpi;
    const int rem = t - img * tpi, ty = rem / ntx;
    y0 = ty * R;
    x0 = (rem - ty * ntx) * kTcOut;
  };
  if (MODE != kFused && warp == kTcEpi) {
    // ---- producer: one TMA copy per half tile (R / 2 + 1 halo rows) ----
    // (one bulk copy per channel group and halo row instead lost by 2.1x)
    if (lane == 0) {
      int q = 0;  // units issued
      bool go = true;
      for (int t = blockIdx.x; go && t < ntiles; t += gridDim.x) {
        int img, y0, x0;
        tile_xy(t, img, y0, x0);
        for (int uu = 0; uu < TU; ++uu, ++q) {
          const int s = q % NU, u = q / NU;
          if (u > 0 && !tc_wait(empty(s), (u - 1) & 1, abort_blk)) {
            go = false;
            break;
          }
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full(s)), "r"(UNIT)
                       : "memory");
          tc_tma4(s_h + s * UNIT, &tm_in, 2 * (x0 - 1), y0 - 1 + UR * uu, img, full(s));
        }
      }
      if (*abort_blk) {  // let the copies in flight land before the block exits
        for (int k = (q > NU ? q - NU : 0); k < q; ++k) {
          const long long t0 = clock64();
          while (!tc_try(full(k % NU), (k / NU) & 1) && clock64() - t0 < kTcWaitCycles) {
          }
        }
      }
    }
  } else if (MODE == kFused && warp >= kTcEpi && warp < kMma) {
    // ---- builders (kFused): the first layer's output over the tile's halo ----
    constexpr int NB = tc_nprod(MODE, R), NBT = 32 * NB;                    // builder warps, threads
    constexpr int XVALS = tc_fx_vals(R), NPRE = (XVALS + NBT - 1) / NBT;  // x values, per builder thread
    static_assert(MODE != kFused || R + 2 == NB, "each builder warp owns a halo row");
    const int bt = tid - 32 * kTcEpi, g = lane >> 2, tq = lane & 3;
    const int bw = warp - kTcEpi;
    uint16_t *xs0 = reinterpret_cast<uint16_t *>(smem + tc_smem(R));  // two parked halos
    constexpr int XS = tc_fx_bytes(R) / 2;
    unsigned char *hs = smem + kTcWBytes;  // generic address of the ring
    auto w1u = [&](int i) { return __bfloat16_as_ushort(__float2bfloat16(w1[i])); };
    uint32_t bf[4][2];  // B fragments: B[k][co] = w1[tap k][co] for k < 9, zero above
    float2 bs[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const int co = 8 * n + g;
      bf[n][0] = pack_u16(w1u((2 * tq) * 32 + co), w1u((2 * tq + 1) * 32 + co));
      bf[n][1] = tq == 0 ? pack_u16(w1u(8 * 32 + co), 0) : 0u;
      bs[n] = make_float2(b1[8 * n + 2 * tq], b1[8 * n + 2 * tq + 1]);
    }
    const int o0 = ((2 * tq) / 3) * kFxP + (2 * tq) % 3, o1 = ((2 * tq + 1) / 3) * kFxP + (2 * tq + 1) % 3;
    constexpr int o8 = 2 * kFxP + 2;
    // barrier of the builders that returns whether any of them saw the abort
    // flag (one decision for all of them)
    auto bar_b_abort = [&]() -> bool {
      uint32_t any;
      asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}"
                   : "=r"(any)
                   : "r"((uint32_t)*abort_blk), "n"(NBT)
                   : "memory");
      return any != 0;
    };
    // this thread's share of tile t's x halo (rows y0 - 2 .., columns x0 - 2
    // ..), left in flight as fp32 until park() rounds and stores it
    auto fetch = [&](int t, float *v) {
      int img, y0, x0;
      tile_xy(t, img, y0, x0);
      const float *src = xin + img * st.xi;
#pragma unroll
      for (int k = 0; k < NPRE; ++k) {
        const int i = bt + NBT * k, r = i / kFxC;
        const int yy = y0 - 2 + r, xx = x0 - 2 + (i - r * kFxC);
        v[k] = (i < XVALS && (unsigned)yy < (unsigned)H && (unsigned)xx < (unsigned)W) ? src[yy * st.xr + xx] : 0.f;
      }
    };
    auto park = [&](const float *v, int b) {
      uint16_t *xs = xs0 + b * XS;
#pragma unroll
      for (int k = 0; k < NPRE; ++k) {
        const int i = bt + NBT * k, r = i / kFxC;
        if (i < XVALS) xs[r * kFxP + (i - r * kFxC)] = __bfloat16_as_ushort(__float2bfloat16(v[k]));
      }
    };
    float v[NPRE];
    if ((int)blockIdx.x < ntiles) {
      fetch(blockIdx.x, v);
      park(v, 0);
    }
    int k = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++k) {
      const int tn = t + gridDim.x;
      if (tn < ntiles) fetch(tn, v);  // in flight while this tile is built
      const int q = k * TU + bw / UR, s = q % NU, u = q / NU;
      if (u > 0) tc_wait(empty(s), (u - 1) & 1, abort_blk);
      // this tile's halo is parked, and every builder is done with the other one
      if (bar_b_abort()) break;
      int img, y0, x0;
      tile_xy(t, img, y0, x0);
      // halo row bw in channel group 0; srow: this lane's 16 bytes of an 8-pixel
      // block for stmatrix, pixel lane % 8 of group lane / 8
      unsigned char *row = hs + s * UNIT + (bw % UR) * kTcHW * 16;
      const uint32_t srow = s_h + s * UNIT + (bw % UR) * kTcHW * 16 + (lane >> 3) * PLANE + (lane & 7) * 16;
      if ((unsigned)(y0 - 1 + bw) >= (unsigned)H) {  // outside the image: the second layer's zero padding
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
          for (int i = lane; i < kTcHW; i += 32)
            *reinterpret_cast<uint4 *>(row + n * PLANE + i * 16) = make_uint4(0u, 0u, 0u, 0u);
      } else {
        const uint16_t *xr = xs0 + (k & 1) * XS + bw * kFxP + g;
#pragma unroll
        for (int i0 = 0; i0 < kTcHW; i0 += 64) {
          uint32_t a[4][4];  // 64 pixels' gathers in flight before the first MMA
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint16_t *p0 = xr + i0 + 16 * i, *p1 = p0 + 8;
            a[i][0] = pack_u16(p0[o0], p0[o1]);
            a[i][1] = pack_u16(p1[o0], p1[o1]);
            a[i][2] = tq == 0 ? (uint32_t)p0[o8] : 0u;
            a[i][3] = tq == 0 ? (uint32_t)p1[o8] : 0u;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float d[4][4];
#pragma unroll
            for (int n = 0; n < 4; ++n) {
              d[n][0] = d[n][2] = bs[n].x;
              d[n][1] = d[n][3] = bs[n].y;
              mma16816(d[n], a[i], bf[n]);
            }
#pragma unroll
            for (int hh = 0; hh < 2; ++hh)  // pixels g (hh = 0) and g + 8
              stm_x4(srow + (i0 + 16 * i + 8 * hh) * 16, cvt_bf16x2<true>(d[0][2 * hh], d[0][2 * hh + 1]),
                     cvt_bf16x2<true>(d[1][2 * hh], d[1][2 * hh + 1]), cvt_bf16x2<true>(d[2][2 * hh], d[2][2 * hh + 1]),
                     cvt_bf16x2<true>(d[3][2 * hh], d[3][2 * hh + 1]));
          }
        }
        // columns outside the image: zero
        const int xw = W - x0 + 1;  // halo pixels from here on lie right of the image
        if (x0 == 0 || xw < kTcHW) {
          __syncwarp();
          if (x0 == 0 && lane < 4) *reinterpret_cast<uint4 *>(row + lane * PLANE) = make_uint4(0u, 0u, 0u, 0u);
          for (int i = xw + (lane >> 2); i < kTcHW; i += 8)
            *reinterpret_cast<uint4 *>(row + (lane & 3) * PLANE + i * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_arrive(full(s));
      if (tn < ntiles) park(v, (k + 1) & 1);
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == kMma) {
    // ---- MMA issuer ----
    if (elect_one()) {
      int k = 0;
      for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++k) {
        const int b = k & 1, ub = k >> 1;
        if (ub > 0 && !tc_wait(tempty(b), (ub - 1) & 1, abort_blk)) break;
        // descriptors differ only in their start-address field: one add per MMA
        // (fully unrolled, the offsets are constants; a single thread issues
        // all of them, so per-MMA arithmetic would bound the tile)
        const uint64_t b0d = umma_desc(s_w, WCG, 128);
        const uint32_t d0 = tmem + b * BUF;
        bool got = true;
#pragma unroll
        for (int uu = 0; uu < TU; ++uu) {
          const int q = k * TU + uu, s = q % NU;
          if (!tc_wait(full(s), (q / NU) & 1, abort_blk)) {
            got = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t a0 = umma_desc(s_h + s * UNIT, PLANE, 128);
#pragma unroll
          for (int hh = 0; hh < UR; ++hh) {
            // output rows h - j for j in [j0, j1] (those inside the tile)
            const int h = UR * uu + hh, j0 = h > R - 1 ? h - (R - 1) : 0, j1 = h < 2 ? h : 2;
            const uint32_t idesc = tc_idesc(NCO * (j1 - j0 + 1));
            const uint32_t d = d0 + (uint32_t)((R - 1 - h + j0) * NCO);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
              for (int ks = 0; ks < 2; ++ks) {
                const uint64_t ad = a0 + (uint64_t)((2 * ks * PLANE + (hh * kTcHW + dx) * 16) >> 4);
                const uint64_t bd = b0d + (uint64_t)((dx * WDX + 2 * ks * WCG + j0 * NCO * 16) >> 4);
                asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                             "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d), "l"(ad),
                             "l"(bd), "r"(idesc), "r"(1u));
              }
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty(s))
                       : "memory");
        }
        if (!got) break;
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tfull(b))
                     : "memory");
      }
    }
  } else {
    // ---- epilogue: warps 0 .. kTcEpi-1, one accumulator row (pixel) per thread ----
    constexpr int RE = R * 4 / kTcEpi;  // output rows per epilogue warp
    const int lq = warp & 3, r0 = (warp >> 2) * RE;
    const uint32_t lanes = (uint32_t)(lq * 32) << 16;
    const long long HWp = (long long)H * W;
    // backward-data: this pixel's sign bits in the rows of a tile, loaded a tile ahead
    auto load_bits = [&](int t, uint32_t *m) {
      int img, y0, x0;
      tile_xy(t, img, y0, x0);
      const int px = lq * 32 + lane, xx = px < kTcOut ? x0 + px : W;
#pragma unroll
      for (int i = 0; i < RE; ++i)
        m[i] = (y0 + r0 + i < H && xx < W) ? bits[img * HWp + (long long)(y0 + r0 + i) * W + xx] : 0u;
    };
    uint32_t sb[RE] = {}, sb_n[RE] = {};
    if (MODE == kBackData && (int)blockIdx.x < ntiles) load_bits(blockIdx.x, sb_n);
    int k = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++k) {
      const int b = k & 1, ub = k >> 1;
      int img, y0, x0;
      tile_xy(t, img, y0, x0);
      if (MODE == kBackData) {
#pragma unroll
        for (int i = 0; i < RE; ++i) sb[i] = sb_n[i];
        if (t + gridDim.x < ntiles) load_bits(t + gridDim.x, sb_n);
      }
      const int px = lq * 32 + lane, xx = px < kTcOut ? x0 + px : W;  // MMA rows 126, 127: no pixel
      float rs[RE];     // last layer: this pixel's residual input, loaded while the MMAs run
      if (MODE == kLast) {
#pragma unroll
        for (int i = 0; i < RE; ++i)
          rs[i] = (y0 + r0 + i < H && xx < W) ? xin[img * st.xi + (y0 + r0 + i) * st.xr + xx] : 0.f;
      }
      const bool ok = tc_wait(tfull(b), ub & 1, abort_blk);
      if (__any_sync(0xffffffffu, !ok)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if constexpr (MODE == kLast) {
#pragma unroll
        for (int rr = r0; rr < r0 + RE; ++rr) {
          const uint32_t ta = tmem + lanes + b * BUF + (R - 1 - rr) * NCO;
          const float v0 = tmem_ld1(ta);
          tmem_zero1(ta);  // channel 0 only: the padding channels never leave zero
          const int yy = y0 + rr;
          if (yy < H && xx < W) out_f[img * st.yi + yy * st.yr + xx] = rs[rr - r0] + v0 + s_bias[0];
        }
      } else {
#pragma unroll(MODE == kBackData ? RE : 1)
        for (int i = 0; i < RE; ++i) {
          const int rr = r0 + i;
          float v[32];
          const uint32_t ta = tmem + lanes + b * BUF + (R - 1 - rr) * NCO;
          tmem_ld32(ta, v);
          tmem_zero32(ta);  // the next tile in this buffer accumulates from zero
          const int yy = y0 + rr;
          if (yy < H && xx < W) {
            const long long pix = (long long)yy * W + xx;
            if (kHid) {
#pragma unroll
              for (int c = 0; c < 32; ++c) v[c] = fmaxf(v[c] + s_bias[c], 0.f);
            }
            uint32_t w = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t pk[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                pk[e] = cvt_bf16x2<false>(v[q * 8 + 2 * e], v[q * 8 + 2 * e + 1]);
                if (MODE == kBackData) pk[e] &= spread(sb[i], 4 * q + e);
              }
              reinterpret_cast<uint4 *>(out)[((long long)img * 4 + q) * HWp + pix] =
                  make_uint4(pk[0], pk[1], pk[2], pk[3]);
              if (MODE == kHidden && bits) {
#pragma unroll
                for (int e = 0; e < 4; ++e) w |= positive(pk[e]) & (0x00010001u << (4 * q + e));
              }
            }
            if (MODE == kHidden && bits) bits[img * HWp + pix] = w;
          }
        }
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      tc_arrive(tempty(b));
    }
  }
  __syncthreads();
  if (tid == 0 && *abort_blk) atomicExch(err, 1);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == kMma) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS));
}

// ldmatrix of four 8 x 8 bf16 matrices, transposed (rows given by lanes 8j .. 8j + 7).
__device__ __forceinline__ void ldsm_x4_t(uint32_t *r, const void *smem_row) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem_row);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(sa));
}

// Weight and bias gradients of the 32 -> 32 layers on the 5th-generation
// tensor cores:
//   dW[dy][dx][co][ci] = sum_p dz[co][p] x[ci][p + (dy - 1, dx - 1)],   db[co] = sum_p dz[co][p].
// Tiles of kWtR rows x kWtC pixels of x; two tensor copies stage its rows (with
// a pixel on either side) and dz's (with a row on either side) as they lie in
// memory, [row][channel group][pixel][8 channels].  That is the MN-major
// operand layout without a swizzle: 8 pixels of a group are a core matrix
// (pixels K, channels MN; 128 contiguous bytes), the next 8 pixels follow, and the
// channel groups of consecutive rows are equally far apart, so one operand may
// span several rows.  An MMA takes four dz rows (M = 4 x 32 channels) against two
// x rows (N = 2 x 32) over 16 pixels (K); the three horizontal taps move x's start by a
// pixel and have accumulators of their own:
//   D_dx[32 j + co][32 i + ci] = sum dz[co][row y - 1 + j][px] x[ci][row y + i][px + dx - 1],
// the tap dy = 2 + i - j for j - i in 0..2; the two other row pairs are not used.
// Three stages: warp 4 copies, one thread of warp 5 issues the MMAs, warps 0-3 (one
// channel group each) sum dz over the tile's own rows for db.  At the end warps 0-3 add
// the two row pairs of each tap in shared memory and the block adds
// them to dW, once.  Bound by DRAM and, close behind, the operands' shared-memory reads
// (6 KB per MMA, 48 cycles): 8 x 512^2 takes 46 us (268 MB: 5.8 TB/s) where staging through registers into swizzled
// pixel-major rows, with two block barriers a tile, took 95.
// Every wait is bounded; a block that gives up flags the error word.
constexpr int kWtR = 8, kWtC = 64, kWtXP = kWtC + 2;        // x rows, pixels per row, staged x pixels per row
constexpr int kWtXRow = 4 * kWtXP * 16, kWtZRow = 4 * kWtC * 16;  // bytes of a staged x, dz row
constexpr int kWtXB = kWtR * kWtXRow, kWtZB = (kWtR + 2) * kWtZRow;  // staged x, dz bytes
constexpr int kWtStage = kWtXB + kWtZB, kWtStages = 3;
constexpr size_t kWtSmem = kWtStages * (size_t)kWtStage + 1024;
static_assert(kWtXB % 128 == 0 && kWtZB % 128 == 0, "the copies land on 128 bytes");
static_assert(kWtSmem <= 227 * 1024, "the stages must fit in shared memory");
static_assert(9 * 32 * 33 * 4 <= kWtStages * kWtStage, "the taps' sums reuse the stages");
// kind::f16, fp32 accumulator, bf16 A and B, both MN-major, N = 64, M = 128
constexpr uint32_t kWtIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
constexpr int kWtThreads = 192;

__device__ __forceinline__ void wt_copy(uint32_t dst, const CUtensorMap *tm, int c0, int y, int img, uint32_t bar) {
  // coordinates (8-byte element along the row, group 0, y, image)
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(0), "r"(y), "r"(img), "r"(bar)
      : "memory");
}

__global__ void __launch_bounds__(kWtThreads, 1) k_conv_wgrad_tc(const __grid_constant__ CUtensorMap tm_x,
                                                                 const __grid_constant__ CUtensorMap tm_z,
                                                                 float *__restrict__ dw, float *__restrict__ db,
                                                                 int nimg, int H, int W, int *err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[2 * kWtStages + 1];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ntx = (W + kWtC - 1) / kWtC, tpi = ntx * ((H + kWtR - 1) / kWtR), ntiles = tpi * nimg;
  const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(s_bar);
  auto full = [&](int i) { return bar0 + 8u * i; };
  auto empty = [&](int i) { return bar0 + 8u * (kWtStages + i); };
  const uint32_t done = bar0 + 8u * (2 * kWtStages);
  volatile int *abort_blk = &s_abort;
  if (tid == 0) {
    s_abort = 0;
    for (int i = 0; i < kWtStages; ++i) {
      tc_mbar_init(full(i), 1);
      tc_mbar_init(empty(i), 5);  // the MMAs and the four warps that sum dz
    }
    tc_mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(
        (uint32_t)__cvta_generic_to_shared(&s_tmem)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
  griddep_wait();
  griddep_launch();
  float bsum[8];  // warps 0-3: channels 8 warp .. 8 warp + 7
#pragma unroll
  for (int c = 0; c < 8; ++c) bsum[c] = 0.f;
  if (warp == 4) {
    if (lane == 0) {
      int k = 0;
      for (int tt = blockIdx.x; tt < ntiles; tt += gridDim.x, ++k) {
        const int s = k % kWtStages, u = k / kWtStages;
        if (u > 0 && !tc_wait(empty(s), (u - 1) & 1, abort_blk)) break;
        const int ts = ntiles - 1 - tt;  // from the last tile, which the kernel before wrote last
        const int img = ts / tpi, rem = ts - img * tpi, ty = rem / ntx;
        const int y0 = ty * kWtR, x0 = (rem - ty * ntx) * kWtC;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full(s)), "r"(kWtStage)
                     : "memory");
        wt_copy(base + s * kWtStage, &tm_x, 2 * (x0 - 1), y0, img, full(s));
        wt_copy(base + s * kWtStage + kWtXB, &tm_z, 2 * x0, y0 - 1, img, full(s));
      }
      if (*abort_blk) {  // let the copies in flight land before the block exits
        for (int i = (k > kWtStages ? k - kWtStages : 0); i < k; ++i) {
          const long long t0 = clock64();
          while (!tc_try(full(i % kWtStages), (i / kWtStages) & 1) && clock64() - t0 < kTcWaitCycles) {
          }
        }
      }
    }
  } else if (__shfl_sync(0xffffffffu, warp, 0) == 5) {
    if (elect_one()) {
      int k = 0;
      for (int tt = blockIdx.x; tt < ntiles; tt += gridDim.x, ++k) {
        const int s = k % kWtStages;
        if (!tc_wait(full(s), (k / kWtStages) & 1, abort_blk)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t X = base + s * kWtStage, Z = X + kWtXB;
        // leading offset: the next 8 pixels; stride offset: the next channel group
        const uint64_t a0 = umma_desc(Z, 128, kWtC * 16), b0 = umma_desc(X, 128, kWtXP * 16);
#pragma unroll
        for (int r = 0; r < kWtR; r += 2)
#pragma unroll
          for (int c = 0; c < kWtC; c += 16)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              const uint64_t ad = a0 + (uint64_t)((r * kWtZRow + c * 16) >> 4);
              const uint64_t bd = b0 + (uint64_t)((r * kWtXRow + (c + dx) * 16) >> 4);
              const uint32_t acc = (k > 0 || r > 0 || c > 0) ? 1u : 0u;
              asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                           "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem + 64 * dx),
                           "l"(ad), "l"(bd), "r"(kWtIdesc), "r"(acc));
            }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty(s))
                     : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(done)
                   : "memory");
      const long long t0 = clock64();  // whatever ended the loop, the MMAs issued finish first
      while (!tc_try(done, 0)) {
        if (clock64() - t0 > kTcWaitCycles) {
          *abort_blk = 1;
          break;
        }
      }
    }
  } else {
    int k = 0;
    for (int tt = blockIdx.x; tt < ntiles; tt += gridDim.x, ++k) {
      const int s = k % kWtStages;
      const bool got = tc_wait(full(s), (k / kWtStages) & 1, abort_blk);
      if (__any_sync(0xffffffffu, !got)) break;
      // dz of the tile's own rows (staged rows 1 .. kWtR), two pixels per thread and row
      const unsigned char *z = smem + s * kWtStage + kWtXB + kWtZRow + (warp * kWtC + lane) * 16;
      float t8[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) t8[c] = 0.f;
#pragma unroll 4
      for (int r = 0; r < kWtR; ++r) {
        static_assert(kWtC == 64, "two pixels of a row per lane");
        const uint4 q[2] = {*reinterpret_cast<const uint4 *>(z + r * kWtZRow),
                            *reinterpret_cast<const uint4 *>(z + r * kWtZRow + 512)};
        const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(q);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __bfloat1622float2(h2[e]), g = __bfloat1622float2(h2[4 + e]);
          t8[2 * e] += f.x + g.x;
          t8[2 * e + 1] += f.y + g.y;
        }
      }
      __syncwarp();
      if (lane == 0) tc_arrive(empty(s));
#pragma unroll
      for (int c = 0; c < 8; ++c) bsum[c] += t8[c];
    }
  }
  __syncthreads();  // the MMAs are done, or the block gave up
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool ok = !s_abort;
  // lane = co, column 64 dx + 32 i + ci; the stages are free
  float *s_w = reinterpret_cast<float *>(smem);  // [tap][co][33]
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    if (ok && warp >= i && warp < 3 + i) {
      const int dyy = 2 + i - warp;
#pragma unroll 1
      for (int dx = 0; dx < 3; ++dx) {
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + 64 * dx + 32 * i, v);
        float *o = s_w + ((3 * dyy + dx) * 32 + lane) * 33;
#pragma unroll
        for (int c = 0; c < 32; ++c) o[c] = i == 0 ? v[c] : o[c] + v[c];
      }
    }
    __syncthreads();
  }
  if (ok) {
    for (int e = tid; e < 9 * 32 * 32; e += kWtThreads) atomicAdd(dw + e, s_w[(e >> 5) * 33 + (e & 31)]);
    if (warp < 4) {
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        float v = bsum[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(db + 8 * warp + c, v);
      }
    }
  }
  if (!ok && tid == 0) atomicExch(err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 5) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem));
}

// Weight and bias gradients of the two one-channel end layers, without
// widening the one channel to 32:
//   first layer:  dW1[tap][co] = sum_p dz1[co][p] x0[p + off(tap)],   db1[co] = sum_p dz1[co][p]
//   last layer:   dW5[tap][ci] = sum_q dy[q - off(tap)] x4[ci][q],    db5 = sum_q dy[q]
// (the last layer's sum re-indexed by q = p + off(tap); the zero padding
// makes both sums run over the image).  Each is a GEMM over the pixels,
// D[tap][c] = sum_p A[tap][p] B[p][c], on mma.sync m16n8k16: M = the 9 taps
// (row 9 all ones for db1, rows 10-15 zero), N = the 32 channels, K = 16
// pixels of a row.  A is the im2col of the one-channel image u (x0, or dy
// rounded to bf16), gathered from its staged halo straight into the A
// fragments; B is the 32-channel operand v (dz1, or x4), staged as it lies
// in global memory (channel-group planar) by 16-byte cp.async copies and read
// with ldmatrix.trans.  db5 is the centre tap's row times a column of ones.
// Persistent blocks of 4 warps walk tiles of 4 rows x 128 pixels (one warp
// per row), double-buffered: tile k + 1's copies and halo loads are in flight
// while tile k is multiplied.  A block sums its warps' partial results in
// shared memory and adds them to the fp32 gradient once.
constexpr int kW1R = 4, kW1C = 128;                       // tile rows, columns
constexpr int kW1HW = kW1C + 2, kW1HP = (kW1R + 2) * kW1HW;  // halo columns, halo values
constexpr int kW1P = 144;                                 // halo row pitch (conflict-free gathers)
constexpr int kW1Pre = (kW1HP + 127) / 128;               // halo values per thread
constexpr int kW1V = 4 * kW1R * kW1C * 8;                 // bf16 of a staged v tile: [group][row][px][8]
constexpr int kW1Red = 9 * 32 + 32;                       // dW [tap][32], then db
constexpr size_t kW1Smem = sizeof(__nv_bfloat16) * 2 * kW1V + sizeof(uint16_t) * 2 * (kW1R + 2) * kW1P +
                           sizeof(float) * kW1Red;

__device__ __forceinline__ uint16_t to_bf16_bits(float v) { return __bfloat16_as_ushort(__float2bfloat16(v)); }
__device__ __forceinline__ uint16_t to_bf16_bits(__nv_bfloat16 v) { return __bfloat16_as_ushort(v); }

template <bool kFirst, typename TU>
__global__ void __launch_bounds__(128) k_conv_wgrad1(const TU *__restrict__ u, const __nv_bfloat16 *__restrict__ v,
                                                     float *__restrict__ dw, float *__restrict__ db, int nimg, int H,
                                                     int W) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  __nv_bfloat16 *s_v = reinterpret_cast<__nv_bfloat16 *>(s_raw);                  // [2][kW1V]
  uint16_t *s_u = reinterpret_cast<uint16_t *>(s_v + 2 * kW1V);                     // [2][(kW1R + 2) * kW1P]
  float *s_red = reinterpret_cast<float *>(s_u + 2 * (kW1R + 2) * kW1P);            // [kW1Red]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int lj = lane >> 3, lr = lane & 7;  // ldmatrix: matrix and row of this lane's address
  const int ntx = (W + kW1C - 1) / kW1C, tpi = ntx * ((H + kW1R - 1) / kW1R), ntiles = tpi * nimg;
  const long long HWp = (long long)H * W;
  for (int i = tid; i < kW1Red; i += 128) s_red[i] = 0.f;
  griddep_wait();
  griddep_launch();
  // halo offsets of this lane's A rows: tap g, and tap 8 (g = 0); the last
  // layer reads u at q - off(tap), the mirrored tap
  const int tg = kFirst ? g : 8 - g;
  const int oT = (tg / 3) * kW1P + tg % 3, o8 = kFirst ? 2 * kW1P + 2 : 0;
  const uint32_t ones = 0x3F803F80u;  // bf16 1.0 pair
  auto origin = [&](int tt, int &img, int &y0, int &x0) {
    img = tt / tpi;
    const int rem = tt - img * tpi, ty = rem / ntx;
    y0 = ty * kW1R;
    x0 = (rem - ty * ntx) * kW1C;
  };
  auto stage_v = [&](int img, int y0, int x0, int b) {
    __nv_bfloat16 *dst = s_v + b * kW1V;
#pragma unroll 4
    for (int i = tid; i < 4 * kW1R * kW1C; i += 128) {
      const int n = i / (kW1R * kW1C), r = (i / kW1C) % kW1R, px = i % kW1C;
      const bool ok = y0 + r < H && x0 + px < W;
      const __nv_bfloat16 *src = ok ? v + (((long long)img * 4 + n) * HWp + (long long)(y0 + r) * W + x0 + px) * 8 : v;
      cp_async16((uint32_t)__cvta_generic_to_shared(dst + (size_t)i * 8), src, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto fetch_u = [&](int img, int y0, int x0, uint16_t *h) {
    const TU *src = u + (long long)img * HWp;
#pragma unroll
    for (int k = 0; k < kW1Pre; ++k) {
      const int i = tid + 128 * k, r = i / kW1HW;
      const int yy = y0 + r - 1, xx = x0 + (i - r * kW1HW) - 1;
      h[k] = (i < kW1HP && (unsigned)yy < (unsigned)H && (unsigned)xx < (unsigned)W)
                 ? to_bf16_bits(src[(long long)yy * W + xx])
                 : (uint16_t)0;
    }
  };
  auto park_u = [&](const uint16_t *h, int b) {
#pragma unroll
    for (int k = 0; k < kW1Pre; ++k) {
      const int i = tid + 128 * k, r = i / kW1HW;
      if (i < kW1HP) s_u[b * (kW1R + 2) * kW1P + r * kW1P + (i - r * kW1HW)] = h[k];
    }
  };
  float acc[4][4], accb[4];
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    accb[n] = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[n][r] = 0.f;
  }
  uint16_t h[kW1Pre];
  int img = 0, y0 = 0, x0 = 0;
  if ((int)blockIdx.x < ntiles) {
    origin(blockIdx.x, img, y0, x0);
    stage_v(img, y0, x0, 0);
    fetch_u(img, y0, x0, h);
    park_u(h, 0);
  }
  int b = 0;
  for (int tt = blockIdx.x; tt < ntiles; tt += gridDim.x, b ^= 1) {
    const int tn = tt + gridDim.x;
    int img_n = 0, y0_n = 0, x0_n = 0;
    if (tn < ntiles) {
      origin(tn, img_n, y0_n, x0_n);
      stage_v(img_n, y0_n, x0_n, b ^ 1);
      fetch_u(img_n, y0_n, x0_n, h);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();  // tile tt's v and u are staged
    if (y0 + warp < H) {
      const uint16_t *ur = s_u + b * (kW1R + 2) * kW1P + warp * kW1P + 2 * t;
      const __nv_bfloat16 *vr = s_v + b * kW1V + warp * kW1C * 8;
      const int nx = min(kW1C, W - x0);
#pragma unroll 2
      for (int c0 = 0; c0 < nx; c0 += 16) {
        uint32_t a[4];
        a[0] = pack_u16(ur[c0 + oT], ur[c0 + oT + 1]);
        a[2] = pack_u16(ur[c0 + oT + 8], ur[c0 + oT + 9]);
        const uint32_t r8a = pack_u16(ur[c0 + o8], ur[c0 + o8 + 1]), r8b = pack_u16(ur[c0 + o8 + 8], ur[c0 + o8 + 9]);
        const uint32_t rone = kFirst && g == 1 ? ones : 0u;
        a[1] = g == 0 ? r8a : rone;
        a[3] = g == 0 ? r8b : rone;
        uint32_t bf[4][2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {  // channel groups 2q, 2q + 1; pixels 0-7 | 8-15
          uint32_t r4[4];
          ldsm_x4_t(r4, vr + ((2 * q + (lj >> 1)) * kW1R * kW1C + c0 + (lj & 1) * 8 + lr) * 8);
          bf[2 * q][0] = r4[0];
          bf[2 * q][1] = r4[1];
          bf[2 * q + 1][0] = r4[2];
          bf[2 * q + 1][1] = r4[3];
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) mma16816(acc[n], a, bf[n]);
        if (!kFirst) {
          const uint32_t bo[2] = {ones, ones};
          mma16816(accb, a, bo);
        }
      }
    }
    if (tn < ntiles) {
      park_u(h, b ^ 1);
      img = img_n;
      y0 = y0_n;
      x0 = x0_n;
    }
    __syncthreads();  // buffer b is refilled by the copies two tiles on
  }
  // D rows: tap g (acc[n][0..1]) and row g + 8 (acc[n][2..3]): tap 8 for
  // g = 0, the ones row (db1) for g = 1; columns 8n + 2t, 8n + 2t + 1
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const int c = 8 * n + 2 * t;
    atomicAdd(&s_red[g * 32 + c], acc[n][0]);
    atomicAdd(&s_red[g * 32 + c + 1], acc[n][1]);
    if (g == 0 || (kFirst && g == 1)) {
      atomicAdd(&s_red[(8 + g) * 32 + c], acc[n][2]);
      atomicAdd(&s_red[(8 + g) * 32 + c + 1], acc[n][3]);
    }
  }
  if (!kFirst && g == 4 && t == 0) atomicAdd(&s_red[9 * 32], accb[0]);  // centre tap x ones: db5
  __syncthreads();
  for (int i = tid; i < 9 * 32; i += 128) atomicAdd(dw + i, s_red[i]);
  if (kFirst) {
    if (tid < 32) atomicAdd(db + tid, s_red[9 * 32 + tid]);
  } else if (tid == 0) {
    atomicAdd(db, s_red[9 * 32]);
  }
}

// fp32 master weights -> bf16 compute weights of the training step: the first
// layer's as they are (the other forward layers round their own), and layers
// 2 .. 5 mirrored and transposed for the backward-data pass, [t][co][ci] ->
// [8 - t][ci][co].
__global__ void k_prep_weights(const float *__restrict__ prm, __nv_bfloat16 *__restrict__ wf, __nv_bfloat16 *__restrict__ wb) {
  const int offs[4] = {kW2, kW3, kW4, kW5};
  const int cout[4] = {C, C, C, 1};
  const int i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  griddep_wait();
  griddep_launch();
  for (int i = i0; i < 9 * C; i += step) wf[i] = __float2bfloat16(prm[kW1 + i]);
  for (int l = 0; l < 4; ++l) {
    const int n = 9 * C * cout[l];
    for (int i = i0; i < n; i += step) {
      const int ci = i % C, co = (i / C) % cout[l], t = i / (C * cout[l]);
      wb[offs[l] + ((8 - t) * C + ci) * cout[l] + co] = __float2bfloat16(prm[offs[l] + i]);
    }
  }
}

// loss = mean((y - t)^2) (fp64 accumulate); dy = 2 (y - t) / n
__global__ void k_mse(const float *__restrict__ y, const float *__restrict__ t, long long n, float *__restrict__ dy,
                      double *loss) {
  griddep_wait();
  griddep_launch();
  double acc = 0.0;
#pragma unroll 4
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    if (dy) dy[i] = 2.f * d / (float)n;
    acc += (double)d * d;
  }
  // one atomic per block (atomics of every warp on one address serialise)
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) atomicAdd(loss, acc / (double)n);
  }
}

// Adam (Kingma & Ba 2015) with bias correction.
__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  griddep_wait();
  griddep_launch();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

template <int R>
void tc_attr() {
  cudaFuncSetAttribute(k_conv_tc<kHidden, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(R));
  cudaFuncSetAttribute(k_conv_tc<kBackData, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(R));
  cudaFuncSetAttribute(k_conv_tc<kLast, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(R));
  cudaFuncSetAttribute(k_conv_tc<kFused, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem_mode(kFused, R));
}

void set_attrs() {
  static bool done = false;
  if (done) return;
  tc_attr<kTcR>();
  tc_attr<kTcRs>();
  cudaFuncSetAttribute(k_conv_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWtSmem);
  cudaFuncSetAttribute(k_conv_wgrad1<false, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kW1Smem);
  cudaFuncSetAttribute(k_conv_wgrad1<true, __nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kW1Smem);
  done = true;
}

// Persistent grid of the one-channel weight-gradient kernel (attributes set by set_attrs).
template <bool kFirst, typename TU>
int grid_wgrad1(int nimg, int H, int W) {
  static int slots = 0;
  if (!slots) {
    int sms = 152, per = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_conv_wgrad1<kFirst, TU>, 128, kW1Smem);
    slots = sms * (per > 0 ? per : 1);
  }
  const long long tiles = (long long)((W + kW1C - 1) / kW1C) * ((H + kW1R - 1) / kW1R) * nimg;
  return (int)(tiles < slots ? tiles : slots);
}

// Persistent grid of the one-channel kernel: its resident blocks, at most one per tile.
template <int MODE>
int grid_1to32(int nimg, int H, int W) {
  static int slots = 0;
  if (!slots) {
    int sms = 152, per = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_conv_1to32<MODE>, 256, 0);
    slots = sms * (per > 0 ? per : 1);
  }
  const long long tiles = (long long)((W + kM1C - 1) / kM1C) * ((H + kM1R - 1) / kM1R) * nimg;
  return (int)(tiles < slots ? tiles : slots);
}


int grid_of(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 152 * 16 ? 152 * 16 : b));
}

// Workspace layout (bytes): bf16 first-layer weights, bf16 weights bwd, x (bf16),
// four hidden activations (bf16, 32 ch), two 32-channel gradient buffers
// (bf16) and the activations' sign bits.
struct Ws {
  __nv_bfloat16 *wf, *wb, *x0, *act[4], *dz[2];
  uint32_t *bits[4];
  size_t bytes;
};

Ws carve(void *ws, long long npx) {
  size_t at = 0;
  auto take = [&](size_t b) {
    char *p = static_cast<char *>(ws) + at;
    at += (b + 255) / 256 * 256;
    return reinterpret_cast<__nv_bfloat16 *>(p);
  };
  const size_t n = (size_t)npx;
  Ws w;
  w.wf = take(2 * kNParams);  // (288 of them are used; the activations 56 KB nearer cost a step of 8 x 512^2 3 us)
  w.wb = take(2 * kNParams);
  w.x0 = take(2 * n);
  for (int l = 0; l < 4; ++l) w.act[l] = take(2 * n * C);
  for (int l = 0; l < 2; ++l) w.dz[l] = take(2 * n * C);
  for (int l = 0; l < 4; ++l) w.bits[l] = reinterpret_cast<uint32_t *>(take(4 * n));
  w.bytes = at;
  return w;
}

size_t ws_bytes(long long npx) { return carve(nullptr, npx).bytes; }

// Error word of the tensor-core kernels' bounded waits (mapped host memory,
// read at the next call).
int *tc_err_host = nullptr, *tc_err_dev = nullptr;

int tc_err() {
  if (!tc_err_host) {
    if (cudaHostAlloc((void **)&tc_err_host, sizeof(int), cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer((void **)&tc_err_dev, tc_err_host, 0) != cudaSuccess) {
      tc_err_host = nullptr;
      return rbc::set_error(RBC_ENOMEM, "error word allocation failed");
    }
    *tc_err_host = 0;
  }
  if (*(volatile int *)tc_err_host) {
    *(volatile int *)tc_err_host = 0;
    return rbc::set_error(RBC_ETIMEOUT, "a tensor-core convolution gave up waiting for its MMAs; results of the "
                                        "calls since the last check are invalid");
  }
  return RBC_OK;
}

// 4-D tensor map over a channel-group planar bf16 activation buffer (32
// channels) seen as 8-byte elements: dims (2 W elements of a row -- two per
// pixel --, y, group, image); box (256 = 128 pixels, by rows, 4 groups, 1).
bool act_map(CUtensorMap *m, const __nv_bfloat16 *buf, int nimg, int H, int W, int by) {
  auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(rbc::tmap_encode_fn());
  if (!fn) return false;
  cuuint64_t dims[4] = {2 * (cuuint64_t)W, (cuuint64_t)H, 4, (cuuint64_t)nimg};
  cuuint64_t strides[3] = {(cuuint64_t)W * 16, (cuuint64_t)W * H * 16, (cuuint64_t)W * H * 64};
  cuuint32_t box[4] = {2 * kTcHW, (cuuint32_t)by, 4, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<__nv_bfloat16 *>(buf), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same buffer with its groups before the rows (the weight gradient's
// operands): dims (2 W elements of a row, group, y, image); box (px pixels, 4
// groups, by rows, 1).
bool rows_map(CUtensorMap *m, const __nv_bfloat16 *buf, int nimg, int H, int W, int px, int by) {
  auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(rbc::tmap_encode_fn());
  if (!fn) return false;
  cuuint64_t dims[4] = {2 * (cuuint64_t)W, 4, (cuuint64_t)H, (cuuint64_t)nimg};
  cuuint64_t strides[3] = {(cuuint64_t)W * H * 16, (cuuint64_t)W * 16, (cuuint64_t)W * H * 64};
  cuuint32_t box[4] = {2 * (cuuint32_t)px, 4, (cuuint32_t)by, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<__nv_bfloat16 *>(buf), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count() {
  static int sms = 0;
  if (!sms) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
  return sms > 0 ? sms : 1;
}

long long tiles_of(int nimg, int H, int W, int R) {
  return (long long)((W + kTcOut - 1) / kTcOut) * ((H + R - 1) / R) * nimg;
}

// Rows per tile: a block's time goes with (tiles per SM) x (R + 2 halo rows),
// so tall tiles win wherever they fill the SMs.  Images of a few hundred rows
// leave SMs idle: one of 200 x 200 takes 27.5 us in 4-row tiles and 30.4 in
// 8-row tiles, while 8 x 512^2 takes 271 and 230.
int tile_rows(int nimg, int H, int W) {
  auto cost = [&](int R) { return (tiles_of(nimg, H, W, R) + sm_count() - 1) / sm_count() * (R + 2); };
  return cost(kTcRs) < cost(kTcR) ? kTcRs : kTcR;
}

template <int MODE, int R>
bool launch_conv_r(const __nv_bfloat16 *in, const void *wt, const float *bias, uint32_t *bits,
                   __nv_bfloat16 *out, int nimg, int H, int W, int rev, cudaStream_t s, float *out_f, const float *x,
                   const Img &st, const float *w1, const float *b1) {
  const long long tiles = tiles_of(nimg, H, W, R);
  const int grid = (int)(tiles < sm_count() ? tiles : sm_count());
  CUtensorMap tin;
  memset(&tin, 0, sizeof tin);  // (the fused mode builds its operand instead of copying it)
  if (MODE != kFused && !act_map(&tin, in, nimg, H, W, tc_ur(R))) return false;
  launch_pdl(k_conv_tc<MODE, R>, dim3(grid), dim3(tc_threads(MODE, R)), tc_smem_mode(MODE, R), s, tin, wt, bias, bits, out,
             out_f, x, st, nimg, H, W, rev, tc_err_dev, w1, b1);
  return true;
}

template <int MODE>
bool launch_conv_tc(const __nv_bfloat16 *in, const void *wt, const float *bias, uint32_t *bits,
                    __nv_bfloat16 *out, int nimg, int H, int W, int rev, cudaStream_t s, float *out_f = nullptr,
                    const float *x = nullptr, const Img &st = Img(), const float *w1 = nullptr,
                    const float *b1 = nullptr) {
  return tile_rows(nimg, H, W) == kTcRs
             ? launch_conv_r<MODE, kTcRs>(in, wt, bias, bits, out, nimg, H, W, rev, s, out_f, x, st, w1, b1)
             : launch_conv_r<MODE, kTcR>(in, wt, bias, bits, out, nimg, H, W, rev, s, out_f, x, st, w1, b1);
}

// One block per SM (its shared memory), at most one per tile.
bool launch_wgrad(const __nv_bfloat16 *x, const __nv_bfloat16 *dz, float *dw, float *db, int nimg, int H, int W,
                  cudaStream_t s) {
  const long long tiles = (long long)((W + kWtC - 1) / kWtC) * ((H + kWtR - 1) / kWtR) * nimg;
  const int grid = (int)(tiles < sm_count() ? tiles : sm_count());
  CUtensorMap tx, tz;
  if (!rows_map(&tx, x, nimg, H, W, kWtXP, kWtR) || !rows_map(&tz, dz, nimg, H, W, kWtC, kWtR + 2)) return false;
  launch_pdl(k_conv_wgrad_tc, dim3(grid), dim3(kWtThreads), kWtSmem, s, tx, tz, dw, db, nimg, H, W, tc_err_dev);
  return true;
}

// The network's forward pass; `keep` stores what the backward pass reads
// (bf16 weights, the bf16 input and the first layer's output: two launches for the first
// two layers, contiguous images); without it the first two layers are one fused launch.
int cnn_forward(const float *params_dev, int nimg, int H, int W, const float *x_dev, float *y_dev, const Img &st,
                void *ws_dev, void *stream, bool keep, const char *who) {
  if (!params_dev || !x_dev || !y_dev || !ws_dev || nimg < 1 || H < 1 || W < 1)
    return rbc::set_error(RBC_EINVAL, who);
  if (int rc = tc_err()) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const long long npx = (long long)nimg * H * W;
  Ws w = carve(ws_dev, npx);
  const float *prm = params_dev;
  set_attrs();
  bool ok_tc = true;
  if (keep) {  // the backward pass reads the first layer's output
    launch_pdl(k_prep_weights, dim3(36), dim3(256), 0, s, prm, w.wf, w.wb);
    launch_pdl(k_conv_1to32<kHidden>, dim3(grid_1to32<kHidden>(nimg, H, W)), dim3(256), 0, s, x_dev, w.x0, w.wf,
               prm + kB1, w.bits[0], w.act[0], nimg, H, W);
    ok_tc = launch_conv_tc<kHidden>(w.act[0], prm + kW2, prm + kB2, w.bits[1], w.act[1], nimg, H, W, 1, s);
  } else {
    ok_tc = launch_conv_tc<kFused>(nullptr, prm + kW2, prm + kB2, nullptr, w.act[1], nimg, H, W, 1, s, nullptr, x_dev,
                                   st, prm + kW1, prm + kB1);
  }
  ok_tc = ok_tc && launch_conv_tc<kHidden>(w.act[1], prm + kW3, prm + kB3, keep ? w.bits[2] : nullptr, w.act[2], nimg,
                                           H, W, 0, s);
  ok_tc = ok_tc && launch_conv_tc<kHidden>(w.act[2], prm + kW4, prm + kB4, keep ? w.bits[3] : nullptr, w.act[3], nimg,
                                           H, W, 1, s);
  ok_tc = ok_tc && launch_conv_tc<kLast>(w.act[3], prm + kW5, prm + kB5, nullptr, nullptr, nimg, H, W, 0, s, y_dev,
                                         x_dev, st);
  if (!ok_tc) return rbc::set_error(RBC_ECUDA, "rbc_cnn_forward: launch failed");
  rbc::add_launches(keep ? 6 : 4);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return rbc::set_error(RBC_ECUDA, cudaGetErrorString(e));
  return RBC_OK;
}

// Strides of contiguous images.
Img packed(int H, int W) { return Img{(long long)H * W, W, (long long)H * W, W}; }

} // namespace

extern "C" {

long long rbc_cnn_param_count(void) { return kNParams; }

long long rbc_cnn_workspace_bytes(int nimg, int H, int W) { return (long long)ws_bytes((long long)nimg * H * W); }

int rbc_cnn_forward(const float *params_dev, int nimg, int H, int W, const float *x_dev, float *y_dev, void *ws_dev,
                    void *stream) {
  return cnn_forward(params_dev, nimg, H, W, x_dev, y_dev, packed(H, W), ws_dev, stream, true,
                     "rbc_cnn_forward: bad arguments");
}

int rbc_cnn_infer(const float *params_dev, int nimg, int H, int W, const float *x_dev, float *y_dev, void *ws_dev,
                  void *stream) {
  return cnn_forward(params_dev, nimg, H, W, x_dev, y_dev, packed(H, W), ws_dev, stream, false,
                     "rbc_cnn_infer: bad arguments");
}

int rbc_cnn_infer_strided(const float *params_dev, int nimg, int H, int W, const float *x_dev, long long x_img,
                          long long x_row, float *y_dev, long long y_img, long long y_row, void *ws_dev,
                          void *stream) {
  if (x_img < 0 || x_row < 0 || y_img < 0 || y_row < 0)
    return rbc::set_error(RBC_EINVAL, "rbc_cnn_infer_strided: negative stride");
  return cnn_forward(params_dev, nimg, H, W, x_dev, y_dev, Img{x_img, x_row, y_img, y_row}, ws_dev, stream, false,
                     "rbc_cnn_infer_strided: bad arguments");
}

int rbc_cnn_backward(const float *params_dev, int nimg, int H, int W, const float *dy_dev, float *grad_dev, void *ws_dev,
                     void *stream) {
  if (!params_dev || !dy_dev || !grad_dev || !ws_dev || nimg < 1 || H < 1 || W < 1)
    return rbc::set_error(RBC_EINVAL, "rbc_cnn_backward: bad arguments");
  if (int rc = tc_err()) return rc;
  set_attrs();
  cudaStream_t s = (cudaStream_t)stream;
  const long long npx = (long long)nimg * H * W;
  Ws w = carve(ws_dev, npx);  // activations from the preceding rbc_cnn_forward

  // layer 5: dW5, db5 from dy; dz4 = conv^T(dy) masked by act4 > 0
  launch_pdl(k_conv_wgrad1<false, float>, dim3(grid_wgrad1<false, float>(nimg, H, W)), dim3(128), kW1Smem, s, dy_dev,
             w.act[3], grad_dev + kW5, grad_dev + kB5, nimg, H, W);
  launch_pdl(k_conv_1to32<kBackData>, dim3(grid_1to32<kBackData>(nimg, H, W)), dim3(256), 0, s, dy_dev, nullptr,
             w.wb + kW5, nullptr, w.bits[3], w.dz[0], nimg, H, W);
  // layers 4, 3, 2: dW from dz; dz below = conv^T(dz) masked
  int cur = 0;
  bool ok_tc = true;
  const int woff[3] = {kW4, kW3, kW2}, boff[3] = {kB4, kB3, kB2};
  for (int l = 0; l < 3; ++l) {
    const int layer_in = 2 - l;  // act index of this layer's input: act3 (l=0) ... act1
    ok_tc = ok_tc && launch_wgrad(w.act[layer_in], w.dz[cur], grad_dev + woff[l], grad_dev + boff[l], nimg, H, W, s);
    ok_tc = ok_tc && launch_conv_tc<kBackData>(w.dz[cur], w.wb + woff[l], nullptr, w.bits[layer_in], w.dz[1 - cur],
                                               nimg, H, W, 0, s);
    cur = 1 - cur;
  }
  // layer 1
  launch_pdl(k_conv_wgrad1<true, __nv_bfloat16>, dim3(grid_wgrad1<true, __nv_bfloat16>(nimg, H, W)), dim3(128), kW1Smem,
             s, w.x0, w.dz[cur], grad_dev + kW1, grad_dev + kB1, nimg, H, W);
  if (!ok_tc) return rbc::set_error(RBC_ECUDA, "rbc_cnn_backward: launch failed");
  rbc::add_launches(9);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return rbc::set_error(RBC_ECUDA, cudaGetErrorString(e));
  return RBC_OK;
}

int rbc_cnn_mse(const float *y_dev, const float *t_dev, long long n, float *dy_dev, double *loss_dev, void *stream) {
  if (!y_dev || !t_dev || !loss_dev || n < 1) return rbc::set_error(RBC_EINVAL, "rbc_cnn_mse: bad arguments");
  // four blocks per SM: each adds its sum to one double, and 2432 such adds took 20 us
  const int most = 4 * sm_count(), grid = grid_of(n) < most ? grid_of(n) : most;
  launch_pdl(k_mse, dim3(grid), dim3(256), 0, (cudaStream_t)stream, y_dev, t_dev, n, dy_dev, loss_dev);
  rbc::add_launches(1);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return rbc::set_error(RBC_ECUDA, cudaGetErrorString(e));
  return RBC_OK;
}

int rbc_cnn_adam(float *params_dev, const float *grad_dev, float *m_dev, float *v_dev, float lr, float b1, float b2,
                 float eps, int step, void *stream) {
  if (!params_dev || !grad_dev || !m_dev || !v_dev || step < 1) return rbc::set_error(RBC_EINVAL, "rbc_cnn_adam: bad arguments");
  // bias corrections formed in fp64: 1 - b2^step cancels badly in fp32 at small steps
  const float c1 = (float)(1.0 - pow((double)b1, (double)step)), c2 = (float)(1.0 - pow((double)b2, (double)step));
  launch_pdl(k_adam, dim3(grid_of(kNParams)), dim3(256), 0, (cudaStream_t)stream, params_dev, grad_dev, m_dev, v_dev,
             kNParams, lr, b1, b2, eps, c1, c2);
  rbc::add_launches(1);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return rbc::set_error(RBC_ECUDA, cudaGetErrorString(e));
  return RBC_OK;
}

} // extern "C"
