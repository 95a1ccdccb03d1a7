// 3x3 convolutions as implicit GEMMs on the tcgen05 tensor cores (paper, Fig. "Convnet activation sampling",
// Sec. 4.2: the conv input is what is sampled; the filter gradient is formed from the sample).  bf16 in,
// float32 accumulation in tensor memory, NHWC, zero padding 1, stride 1.
//
//   forward          M = output pixels (a tile of 128: 32 pooling windows, the four pixels of a window in four
//                    neighbouring accumulator rows), N = Cout (padded to 64), K = 9 Cin taken 64 at a time.  The A
//                    tile is the im2col patch matrix, written K-major into shared memory by the CTA's threads
//                    (no patch matrix ever exists in global memory); B is the filter block.  The epilogue adds the
//                    bias, applies ReLU, packs the four derivative bits of a window and writes the 2x2 average.
//   filter gradient  dW[(tap, ci), co] = sum over pixels of A_hat[pixel + tap, ci] dZ[pixel, co]: M = (tap, ci) in
//                    tiles of 128, N = Cout (padded to 64), K = pixels, split over CTAs; both operands are
//                    MN-major (the contraction index is the slow index of both tensors).  A_hat is the sampled
//                    conv input, expanded from its compact store into a zero-filled NHWC buffer of one layer
//                    (held only while this layer's gradient is formed).  Partial tiles are summed in split order.
//   input gradient   dX[pixel, ci] = sum over (tap, co) of dZ[pixel - tap, co] W[tap, ci, co] (the transposed
//                    convolution, exact): M = input pixels in raster order, N = Cin (padded to 64), K = 9 Cout taken
//                    64 at a time; the A tile is the patch matrix of dZ with the taps mirrored, K-major as in the
//                    forward pass; B is K-major too (for a tap and an input channel the output channels are
//                    contiguous in the filter tensor); the epilogue rounds and writes 64 bytes per row and chunk.
//
// One CTA (no cluster), eight warps: all of them write operand tiles with the 128-byte swizzle the tensor core
// expects (16-byte chunk c of row r lands at chunk c ^ (r & 7)), one elected thread issues tcgen05.mma.cta_group::1
// (M128 N64 K16), two shared-memory stages alternate, the 128 x 64 accumulator takes 64 columns of tensor
// memory.  Every wait is bounded; on expiry the CTA raises RAD_DEV_ETIMEOUT, frees its tensor memory and returns.
#include <algorithm>

#include "common.cuh"
#include "umma.cuh"

namespace rad {
namespace {

constexpr int kCvM = 128, kCvN = 64, kCvK = 64;
constexpr int kCvThreads = 256;
constexpr int kCvPerSm = 4;                      // CTAs that fit an SM: shared memory, 64 registers a thread, 256 tensor-memory columns
constexpr int kCvABytes = kCvM * kCvK * 2;       // 16 KB either way round
constexpr int kCvBBytes = kCvK * kCvN * 2;       // 8 KB
constexpr int kCvStageBytes = kCvABytes + kCvBBytes;

struct ConvTcParams {
  int64_t B;
  int32_t H, W, Cin, Cout;
  const bf16* X;            // forward: conv input; filter gradient: A_hat (zero where dropped), both NHWC dense
  const bf16* Wt;           // 3 x 3 x Cin x Cout
  const float* bias;
  bf16* P;                  // pooled output; input gradient: dX, B x H x W x Cin
  uint32_t* relubits;
  const bf16* dZ;           // B x H x W x Cout
  float* partial;           // splits x (9 Cin) x Cout
  int32_t kblocks_per_split;
  int32_t* dev_status;
  uint64_t wait_limit_ns;
};

struct CvCtl {
  uint64_t done[2];        // the MMAs that read stage s have retired
  uint32_t tmem_base;
  int abort_flag;
};

// 16 bytes of a dense NHWC tensor at pixel (y, x) of the image that starts at T, channel c0 .. c0 + 7, zero outside
__device__ __forceinline__ uint4 cv_load_pixel(const bf16* T, bool in, int y, int x, int H, int W, int C, int c0) {
  if (!in || y < 0 || y >= H || x < 0 || x >= W) return make_uint4(0u, 0u, 0u, 0u);
  return *reinterpret_cast<const uint4*>(T + ((int64_t)y * W + x) * C + c0);
}

// kCvFwd: forward tile `blockIdx.x` (128 output pixels); kCvDw: filter-gradient unit (m tile, split) = blockIdx;
// kCvDx: input-gradient tile `blockIdx.x` (128 input pixels in raster order).
// What bounds these kernels is the chain of a K block: gather (L2 latency), store to shared memory, fence, MMA.  So the
// gather of the next block is in registers before this block's stage is waited for, a block costs one barrier, and all
// of a thread's index arithmetic that does not change from block to block (its pixels in the forward and input
// gradient, its tap and channels in the filter gradient) is done once.  CNN at batch 4096, second / third
// convolution: forward 279 -> 164 / 123 -> 58 us, filter gradient (also 444 instead of 192 CTAs) 855 -> 138 /
// 210 -> 58, input gradient 339 -> 175 / 165 -> 78.
enum { kCvFwd = 0, kCvDw = 1, kCvDx = 2 };
template <int kMode>
__global__ void __launch_bounds__(kCvThreads, kCvPerSm) conv_tc_kernel(const ConvTcParams p) {
  constexpr bool kDw = kMode == kCvDw, kDx = kMode == kCvDx;
  extern __shared__ uint8_t cv_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(cv_raw) + 1023) & ~(uintptr_t)1023);
  CvCtl* ctl = reinterpret_cast<CvCtl*>(smem + 2 * kCvStageBytes);
  volatile int* abort_flag = &ctl->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = p.H, W = p.W, Cin = p.Cin, Cout = p.Cout;
  const int64_t npix = p.B * H * W;
  const int ktaps = 9 * Cin;                          // rows of the filter matrix
  if (tid == 0) {
    for (int s = 0; s < 2; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(umma_smem(&ctl->done[s])), "r"(1u) : "memory");
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(umma_smem(&ctl->tmem_base)), "r"(64u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }

  // what this CTA contracts over
  const int mtile = kDw ? (int)blockIdx.x : 0, split = kDw ? (int)blockIdx.y : 0;
  const int64_t tile = kDw ? 0 : blockIdx.x;
  const int nkb = kDw ? p.kblocks_per_split : ((kDx ? 9 * Cout : ktaps) + kCvK - 1) / kCvK;
  const int64_t kb0 = kDw ? (int64_t)split * p.kblocks_per_split : 0;

  // Patch operand A.  Forward, input gradient: thread = 16-byte chunk cc (k = 8 cc ..) of rows m0 + 32 j, whose pixels
  // stay; K-major.  Filter gradient: thread = chunk cc (eight (tap, ci) indices, which stay) of the pixels k0 + 16 j,
  // which move on by 64 a block; MN-major.
  constexpr int kRowShift = kDw ? 4 : 3;
  const int cc = tid & ((1 << kRowShift) - 1), row0 = tid >> kRowShift;
  const bf16* img[4];                                 // image of the pixel
  int py[4], px[4];
  bool in[4];
  const int C = kDx ? Cout : Cin;                     // channels of the gathered tensor
  const bf16* src = kDx ? p.dZ : p.X;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (kDw) {
      const int64_t pix = kb0 * kCvK + row0 + 16 * j, line = pix / W;
      px[j] = (int)(pix - line * W); py[j] = (int)(line % H);
      img[j] = src + (line / H) * H * W * C;
      in[j] = pix < npix;
    } else if (kDx) {
      const int64_t pix = tile * kCvM + row0 + 32 * j, line = pix / W;
      px[j] = (int)(pix - line * W); py[j] = (int)(line % H);
      img[j] = src + (line / H) * H * W * C;
      in[j] = pix < npix;
    } else {
      // row m = window (tile * 32 + m / 4), pixel m % 4 of it
      const int m = row0 + 32 * j, Wp = W >> 1, Hp = H >> 1;
      const int64_t q = tile * 32 + (m >> 2), line = q / Wp;
      px[j] = 2 * (int)(q - line * Wp) + (m & 1); py[j] = 2 * (int)(line % Hp) + ((m >> 1) & 1);
      img[j] = src + (line / Hp) * H * W * C;
      in[j] = q < npix / 4;
    }
  }
  // the filter gradient's (tap, channels) and its step of 64 pixels
  const int dw_m0 = mtile * kCvM + cc * 8, dw_tap = kDw ? dw_m0 / Cin : 0, dw_c0 = dw_m0 - dw_tap * Cin;
  const int step_x = kCvK % W, step_l = kCvK / W, step_y = step_l % H;
  const int64_t step_img = (int64_t)(step_l / H) * H * W * C, one_img = (int64_t)H * W * C;
  uint4 va[4], vb[2];
  int64_t left = kDw ? npix - kb0 * kCvK - row0 : 0;  // pixels from this thread's first one to the end
  auto gather = [&](int kb) {
    if (kDw) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        va[j] = cv_load_pixel(img[j], left > 16 * j && dw_tap < 9, py[j] + dw_tap / 3 - 1, px[j] + dw_tap % 3 - 1, H, W, C, dw_c0);
        px[j] += step_x; py[j] += step_y; img[j] += step_img;
        if (px[j] >= W) { px[j] -= W; ++py[j]; }
        if (py[j] >= H) { py[j] -= H; img[j] += one_img; }
      }
      left -= kCvK;
      // B: dZ of the pixel, 8 chunks of 8 channels per row
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int k = (tid >> 3) + 32 * j, c = (tid & 7) * 8;
        const int64_t pix = (kb0 + kb) * kCvK + k;
        vb[j] = pix < npix && c < Cout ? *reinterpret_cast<const uint4*>(p.dZ + pix * Cout + c) : make_uint4(0u, 0u, 0u, 0u);
      }
    } else {
      const int k0 = kb * kCvK + cc * 8, tap = k0 / C, c0 = k0 - tap * C, ty = tap / 3, tx = tap - 3 * ty;
      // forward: the tap reads pixel (y + ty - 1, x + tx - 1); input gradient: the output pixel that reached this input
      // pixel through the tap lies at (y - ty + 1, x - tx + 1)
      const int dy = kDx ? 1 - ty : ty - 1, dx = kDx ? 1 - tx : tx - 1;
#pragma unroll
      for (int j = 0; j < 4; ++j) va[j] = cv_load_pixel(img[j], in[j] && tap < 9, py[j] + dy, px[j] + dx, H, W, C, c0);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = (tid >> 3) + 32 * j;
        vb[j] = make_uint4(0u, 0u, 0u, 0u);
        if (kDx) {
          // B: K-major, row n = input channel, k = (tap, co): W[tap, n, co0 .. co0 + 7] is contiguous
          if (tap < 9 && r < Cin) vb[j] = *reinterpret_cast<const uint4*>(p.Wt + ((int64_t)tap * Cin + r) * Cout + c0);
        } else {
          // B: filter rows k (MN-major: Cout contiguous), 8 chunks of 8 channels per row
          const int kg = kb * kCvK + r;
          if (kg < ktaps && cc * 8 < Cout) vb[j] = *reinterpret_cast<const uint4*>(p.Wt + (int64_t)kg * Cout + cc * 8);
        }
      }
    }
  };
  wait_for_previous();                                // behind the tensor memory and all that only needs the parameters
  if (nkb > 0) gather(0);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = ctl->tmem_base;
  let_next_start();

  bool ok = true;
  for (int kb = 0; kb < nkb; ++kb) {
    const int s = kb & 1;
    uint8_t* sA = smem + s * kCvStageBytes;
    uint8_t* sB = sA + kCvABytes;
    // the MMAs of two K blocks ago have read this stage
    if (kb >= 2) ok = umma_wait(umma_smem(&ctl->done[s]), ((kb >> 1) - 1) & 1, abort_flag, p.wait_limit_ns);
    if (ok) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = row0 + (kDw ? 16 : 32) * j;
        if (kDw) *reinterpret_cast<uint4*>(sA + (cc >> 3) * 8192 + r * 128 + (((cc & 7) ^ (r & 7)) << 4)) = va[j];
        else *reinterpret_cast<uint4*>(sA + r * 128 + ((cc ^ (r & 7)) << 4)) = va[j];
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = (tid >> 3) + 32 * j, c = tid & 7;
        *reinterpret_cast<uint4*>(sB + r * 128 + ((c ^ (r & 7)) << 4)) = vb[j];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (!__syncthreads_and(ok ? 1 : 0)) { ok = false; break; }
    if (warp == 0 && elect_one()) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      constexpr uint32_t idesc = umma_idesc(kCvM, kCvN, kDw, !kDx);
      const uint32_t a0 = umma_smem(sA), b0 = umma_smem(sB);
#pragma unroll
      for (int k = 0; k < kCvK / 16; ++k) {
        const uint64_t adesc = kDw ? umma_desc(a0 + k * 2048, 8192, 1024) : umma_desc(a0 + k * 32, 16, 1024);
        const uint64_t bdesc = kDx ? umma_desc(b0 + k * 32, 16, 1024) : umma_desc(b0 + k * 2048, 8192, 1024);
        umma_mma(tmem, adesc, bdesc, idesc, (kb > 0 || k > 0) ? 1u : 0u);
      }
      umma_commit(umma_smem(&ctl->done[s]));
    }
    if (kb + 1 < nkb) gather(kb + 1);
  }
  // the last commit covers every MMA before it
  if (ok && nkb > 0) ok = umma_wait(umma_smem(&ctl->done[(nkb - 1) & 1]), ((nkb - 1) >> 1) & 1, abort_flag, p.wait_limit_ns);
  ok = __syncthreads_and(ok ? 1 : 0) != 0;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok) {
    const int q = warp & 3, chunk = warp >> 2;       // accumulator rows 32 q .. 32 q + 31, columns 32 chunk .. + 31
    const int m = q * 32 + lane;
    uint32_t r[32];
    umma_tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(chunk * 32), r);
    if (kDx) {
      // row m = input pixel, columns = input channels: rounded once, 64 bytes per row and chunk
      const int64_t pix = tile * kCvM + m;
      if (pix < npix) {
        bf16* dst = p.P + pix * Cin + chunk * 32;
#pragma unroll
        for (int j = 0; j < 32; j += 8) {
          if (chunk * 32 + j < Cin) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(r[j + 2 * e]), __uint_as_float(r[j + 2 * e + 1]));
              w[e] = *reinterpret_cast<const uint32_t*>(&h2);
            }
            *reinterpret_cast<uint4*>(dst + j) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      }
    } else if (!kDw) {
      // rows 4 w .. 4 w + 3 are the 2 x 2 window w.  Each lane adds the bias, applies ReLU and rounds for its own pixel;
      // then the four lanes of a window exchange (two rounds of shuffles), so that lane q holds all four pixels of channels
      // 8 q .. 8 q + 7 of the chunk: one word of derivative bits and one 16-byte store of rounded averages.
      const int64_t win = tile * 32 + (m >> 2);
      const int q4 = lane & 3, co0 = chunk * 32 + q4 * 8;
      float a[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const int co = chunk * 32 + j;
        const float z = __uint_as_float(r[j]) + (p.bias != nullptr && co < Cout ? p.bias[co] : 0.0f);
        a[j] = __bfloat162float(__float2bfloat16_rn(fmaxf(z, 0.0f)));       // the activation as the device would hold it
      }
      // round 1, partner lane ^ 1: keep channel blocks q & 1 and 2 + (q & 1) of eight
      float mine[2][8], theirs[2][8];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float lo = a[16 * h + c], hi = a[16 * h + 8 + c];
          mine[h][c] = (q4 & 1) ? hi : lo;
          theirs[h][c] = __shfl_xor_sync(0xffffffffu, (q4 & 1) ? lo : hi, 1);
        }
      // round 2, partner lane ^ 2: keep half q >> 1; then the pixels in order 0 .. 3
      uint32_t word = 0;
      __align__(16) bf16 pooled[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const bool up = (q4 & 2) != 0, odd = (q4 & 1) != 0;
        const float s0 = up ? mine[1][c] : mine[0][c], s1 = up ? theirs[1][c] : theirs[0][c];
        const float t0 = __shfl_xor_sync(0xffffffffu, up ? mine[0][c] : mine[1][c], 2);
        const float t1 = __shfl_xor_sync(0xffffffffu, up ? theirs[0][c] : theirs[1][c], 2);
        const float se = odd ? s1 : s0, so = odd ? s0 : s1, te = odd ? t1 : t0, to = odd ? t0 : t1;     // even, odd pixel of either pair
        const float a0 = up ? te : se, a1 = up ? to : so, a2 = up ? se : te, a3 = up ? so : to;
        word |= ((a0 > 0.0f ? 1u : 0u) | (a1 > 0.0f ? 2u : 0u) | (a2 > 0.0f ? 4u : 0u) | (a3 > 0.0f ? 8u : 0u)) << (4 * c);
        pooled[c] = __float2bfloat16_rn(0.25f * (((a0 + a1) + a2) + a3));
      }
      if (win < npix / 4 && co0 < Cout) {
        *reinterpret_cast<uint4*>(p.P + win * Cout + co0) = *reinterpret_cast<const uint4*>(pooled);
        p.relubits[(win * Cout + co0) >> 3] = word;
      }
    } else {
      const int mg = mtile * kCvM + m;
      if (mg < ktaps) {
        float* dst = p.partial + ((int64_t)split * ktaps + mg) * Cout + chunk * 32;
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          if (chunk * 32 + j < Cout)
            *reinterpret_cast<float4*>(dst + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                              __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && ctl->abort_flag != 0) raise_status(p.dev_status, RAD_DEV_ETIMEOUT);
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(64u) : "memory");
  }
}

// A_hat (B x D, zero where dropped) from a compact store.  different-sample: a thread per keep-bit word writes its 32
// columns, zeros first, so that the buffer needs no clearing of its own (a clear between two kernels costs both of them their
// overlap: 3 us).  same-sample: the buffer is cleared, then a thread per kept entry.
__global__ void __launch_bounds__(256) densify_different_kernel(const bf16* values, const uint32_t* keepbits, const uint32_t* offsets,
                                                                int64_t B, int64_t D, int32_t ncb, int64_t capacity, bf16* out) {
  begin_after_previous();
  const int64_t nwords = ((B + kTileRows - 1) / kTileRows) * ncb * kBitWords;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nwords; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t tile = i / kBitWords;
    const int t = (int)(i - tile * kBitWords), r = t >> 2, w = t & 3;
    const int64_t row = (tile / ncb) * kTileRows + r, col0 = (tile % ncb) * kTileCols + 32 * w;
    if (row >= B || col0 >= D) continue;
    bf16* dst = out + row * D + col0;               // D is a multiple of 64: whole words, 16-byte aligned
#pragma unroll
    for (int j = 0; j < 4; ++j) reinterpret_cast<uint4*>(dst)[j] = make_uint4(0u, 0u, 0u, 0u);
    const uint32_t* tw = keepbits + tile * kTileWords;
    uint32_t word = tw[t];
    int64_t pos = (int64_t)offsets[tile] + ((tw[kBitWords + (r >> 1)] >> (16 * (r & 1))) & 0xffffu);
    for (int q = 0; q < w; ++q) pos += __popc(tw[r * 4 + q]);
    while (word != 0) {
      const int b = __ffs(word) - 1;
      word &= word - 1;
      if (pos < capacity) dst[b] = values[pos];
      ++pos;
    }
  }
}
__global__ void __launch_bounds__(256) densify_same_kernel(const bf16* values, const uint32_t* idx, const int64_t* nnz, int64_t B,
                                                           int64_t D, int64_t ld, bf16* out) {
  begin_after_previous();
  const int64_t k = min(nnz[0], ld);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < B * k; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = i / k, j = i - b * k;
    const uint32_t col = idx[j];
    if (col < (uint32_t)D) out[b * D + col] = values[b * ld + j];
  }
}

constexpr size_t kCvSmem = 2 * kCvStageBytes + sizeof(CvCtl) + 1024;
int g_conv_kernel = RAD_CONV_KERNEL_AUTO;

}  // namespace

bool conv_tensor_allowed() { return g_conv_kernel != RAD_CONV_KERNEL_SIMT; }

// Shapes the tensor-core kernels take: bf16, Cin 16, 32 or 64 (a 64-deep K block is a whole number of taps),
// Cout a multiple of 8 up to 64, even H and W.
bool conv_tc_ok(int dtype, int H, int W, int Cin, int Cout, const void* X, const void* Wt) {
  if (g_conv_kernel == RAD_CONV_KERNEL_SIMT) return false;
  return dtype == RAD_BF16 && (Cin == 16 || Cin == 32 || Cin == 64) && Cout % 8 == 0 && Cout >= 8 && Cout <= kCvN && H % 2 == 0 &&
         W % 2 == 0 && ((uintptr_t)X & 15) == 0 && ((uintptr_t)Wt & 15) == 0;
}

int conv_tc_forward_pool(int64_t B, int H, int W, int Cin, int Cout, const void* X, const void* Wt, const float* bias, void* P,
                         uint32_t* relubits, int32_t* dev_status, cudaStream_t st) {
  ConvTcParams p = {};
  p.B = B; p.H = H; p.W = W; p.Cin = Cin; p.Cout = Cout;
  p.X = static_cast<const bf16*>(X); p.Wt = static_cast<const bf16*>(Wt); p.bias = bias;
  p.P = static_cast<bf16*>(P); p.relubits = relubits; p.dev_status = dev_status; p.wait_limit_ns = wait_limit_ns();
  RAD_CUDA_TRY(cudaFuncSetAttribute(conv_tc_kernel<kCvFwd>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCvSmem));
  const int64_t windows = B * (H / 2) * (W / 2);
  count_launch();
  RAD_TRY(launch_kernel(conv_tc_kernel<kCvFwd>, (unsigned)ceil_div(windows, 32), kCvThreads, kCvSmem, st, p));
  return RAD_OK;
}

// Shapes the input-gradient kernel takes: as above with the channel counts in each other's roles (K runs over
// (tap, co) in chunks of eight output channels, N over the input channels).
bool conv_tc_dx_ok(int dtype, int H, int W, int Cin, int Cout, const void* dZ, const void* Wt, const void* dX) {
  (void)H; (void)W;
  if (g_conv_kernel == RAD_CONV_KERNEL_SIMT) return false;
  return dtype == RAD_BF16 && (Cout == 16 || Cout == 32 || Cout == 64) && Cin % 8 == 0 && Cin >= 8 && Cin <= kCvN &&
         ((uintptr_t)dZ & 15) == 0 && ((uintptr_t)Wt & 15) == 0 && ((uintptr_t)dX & 15) == 0;
}

int conv_tc_input_grad(int64_t B, int H, int W, int Cin, int Cout, const void* dZ, const void* Wt, void* dX, int32_t* dev_status,
                       cudaStream_t st) {
  ConvTcParams p = {};
  p.B = B; p.H = H; p.W = W; p.Cin = Cin; p.Cout = Cout;
  p.dZ = static_cast<const bf16*>(dZ); p.Wt = static_cast<const bf16*>(Wt); p.P = static_cast<bf16*>(dX);
  p.dev_status = dev_status; p.wait_limit_ns = wait_limit_ns();
  RAD_CUDA_TRY(cudaFuncSetAttribute(conv_tc_kernel<kCvDx>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCvSmem));
  count_launch();
  RAD_TRY(launch_kernel(conv_tc_kernel<kCvDx>, (unsigned)ceil_div(B * H * W, kCvM), kCvThreads, kCvSmem, st, p));
  return RAD_OK;
}

// K blocks of 64 pixels per CTA of the filter-gradient kernel, and the splits that follow from it: enough for four
// CTAs on every SM (a K block is a chain of latencies, so CTAs side by side are what hides them), at least four each.
static int conv_tc_splits(int64_t npix, int Cin, int* kblocks_per_split) {
  const int64_t kblocks = ceil_div(npix, kCvK), want = std::max<int64_t>(1, kCvPerSm * 148 / ceil_div(9 * Cin, kCvM));
  const int64_t per = std::max<int64_t>(4, ceil_div(kblocks, want));
  *kblocks_per_split = (int)per;
  return (int)ceil_div(kblocks, per);
}

int64_t conv_tc_weight_grad_workspace(int64_t B, int H, int W, int Cin, int Cout) {
  int per = 0;
  const int splits = conv_tc_splits(B * H * W, Cin, &per);
  return round_up(B * H * W * Cin * 2, 256) + round_up((int64_t)splits * 9 * Cin * Cout * 4, 256) +
         column_sums_workspace(splits, 9 * Cin * Cout);
}

int conv_tc_weight_grad(const rad_store* store, int H, int W, int Cin, int Cout, const void* dZ, float* dW, void* workspace,
                        int64_t workspace_bytes, int32_t* dev_status, cudaStream_t st) {
  const int64_t B = store->B, D = store->D;
  if (workspace == nullptr || workspace_bytes < conv_tc_weight_grad_workspace(B, H, W, Cin, Cout)) return RAD_EWORKSPACE;
  bf16* dense = static_cast<bf16*>(workspace);
  float* partial = reinterpret_cast<float*>(static_cast<char*>(workspace) + round_up(B * D * 2, 256));
  count_launch();
  if (store->variant == RAD_SAME_SAMPLE) {
    RAD_CUDA_TRY(cudaMemsetAsync(dense, 0, (size_t)(B * D * 2), st));
    RAD_TRY(launch_kernel(densify_same_kernel, (unsigned)std::min<int64_t>(ceil_div(B * store->values_ld, 256), 148 * 16), 256, 0, st, static_cast<const bf16*>(store->values), store->offsets, store->nnz, B, D, store->values_ld, dense));
  } else {
    const int32_t ncb = (int32_t)ceil_div(D, kTileCols);
    const int64_t nwords = ceil_div(B, kTileRows) * ncb * kBitWords;
    RAD_TRY(launch_kernel(densify_different_kernel, (unsigned)std::min<int64_t>(ceil_div(nwords, 256), 148 * 16), 256, 0, st, static_cast<const bf16*>(store->values), store->keepbits, store->offsets, B, D, ncb, store->values_capacity, dense));
  }
  ConvTcParams p = {};
  p.B = B; p.H = H; p.W = W; p.Cin = Cin; p.Cout = Cout;
  p.X = dense; p.dZ = static_cast<const bf16*>(dZ); p.partial = partial; p.dev_status = dev_status;
  p.wait_limit_ns = wait_limit_ns();
  const int splits = conv_tc_splits(B * H * W, Cin, &p.kblocks_per_split);
  RAD_CUDA_TRY(cudaFuncSetAttribute(conv_tc_kernel<kCvDw>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCvSmem));
  count_launch();
  RAD_TRY(launch_kernel(conv_tc_kernel<kCvDw>, dim3((unsigned)ceil_div(9 * Cin, kCvM), (unsigned)splits), kCvThreads, kCvSmem, st, p));
  // the splits' partial sums: column sums of a splits x (9 Cin Cout) matrix, in a fixed order
  const int64_t n = (int64_t)9 * Cin * Cout, held = round_up((int64_t)splits * n * 4, 256);
  return column_sums(RAD_F32, splits, n, partial, n, dW, reinterpret_cast<char*>(partial) + held, column_sums_workspace(splits, n), st);
}

}  // namespace rad

extern "C" int rad_set_conv_kernel(int32_t which) {
  if (which != RAD_CONV_KERNEL_AUTO && which != RAD_CONV_KERNEL_SIMT && which != RAD_CONV_KERNEL_TENSOR) return RAD_EINVAL;
  const int prev = rad::g_conv_kernel;
  rad::g_conv_kernel = which;
  return prev;
}
