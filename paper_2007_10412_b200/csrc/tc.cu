// tcgen05 GEMM engine (bf16 in, float32 accumulate in tensor memory) for the four contractions of
// a RAD step on large aligned layers:
//   forward      Z = A W + b                 (exact; Sec. 3: the forward pass is the original graph)
//   input grad   dA = dZ W^T                 (exact; Sec. 4.2)
//   dW, same     dW[idx, :] = A_c^T dZ       (column-compacted dense GEMM; Sec. 4.3 "same sample")
//   dW, diff.    dW = A_hat^T dZ             (A_hat tiles rebuilt in shared memory from keep bits
//                                             and packed values; Sec. 4.2 / 4.3 "different sample")
//
// Every kernel here runs on SM pairs: a cluster of two CTAs, one per SM, persistent, with one
// thread of the even CTA issuing tcgen05.mma.cta_group::2 on operands that both CTAs stage in their
// own shared memory (TMA, 128-byte swizzle, no multicast) through an mbarrier ring.
//   dense kernels    256 x 256 tile per pair, or 128 or 64 columns wide where that makes one wave of
//                    them or the matrix has no more; each CTA keeps two alternating 128 x 256 float32
//                    accumulators in tensor memory, so the epilogue of a tile (bias, activation,
//                    ReLU bits, GELU', TMA stores) runs under the MMAs of the next one.  The input
//                    gradient's epilogue warps make the bias gradient while they wait, where the
//                    K blocks of the tiles hide it.
//   sparse-A kernel  256 x 512 tile per pair (256 or 128 columns where 512 would leave SMs idle);
//                    sixteen "expander" warps per CTA write the A_hat tile of each K block into
//                    shared memory instead of TMA.
// Long dW contractions can be split along K; partial tiles are summed in split order by a second
// kernel, so results are reproducible.
// Every mbarrier wait is bounded: on expiry both CTAs of the pair raise their abort flags, all
// roles leave their loops, the pair meets at a cluster barrier, tensor memory is released, the
// kernel returns and the launch reports RAD_DEV_ETIMEOUT.
#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "store.cuh"

namespace rad {
namespace {

constexpr int BM = 256, BN = 256, BK = 64;
constexpr int kNumSMsDefault = 148;
constexpr int kMaxSplits = 16;
constexpr int kRasterGroup = 16;               // m-tiles per raster group (16 x 4 MB of A panels stay in L2 beside the B panels in flight)

enum AKind { kAK = 0, kAMN = 1, kASparse = 2 };
enum BKind { kBK_ = 0, kBMN = 1 };
// Epilogues: forward pass by activation (RAD_ACT_*), without and with the filling of the next layer's store; input gradient,
// plain or masked by ReLU bits, and times GELU'(z); same-sample dW, transposed.
enum EpiKind { kFwd = 0, kFwdFill = 3, kDx = 6, kDxGelu = 7, kDwT = 8 };
constexpr bool is_forward(int epi) { return epi < kDx; }
constexpr bool is_dx(int epi) { return epi == kDx || epi == kDxGelu; }

struct TcParams {
  int64_t M, N, K;
  const int64_t* N_dev;      // same-sample dW: N = number of kept columns, read on the device
  const uint32_t* keep_cols; // same-sample dW: bit d set = column d of the layer input was kept
  int32_t bn;                // columns of an output tile (forward, input gradient: 64, 128 or 256; sparse A: 128, 256 or 512)
  int32_t splits;            // K splits (1: epilogue writes final results)
  int32_t num_stages;        // of the ring of operand stages
  int32_t comp_depth;        // sparse A: depth of the ring of compressed (index + values) buffers
  // sparse A (different-sample store)
  const bf16* values; const uint32_t* keepbits; const uint32_t* offsets;
  int64_t values_capacity; int32_t ncb; int32_t comp_cap;   // comp_cap: value bytes per half-stage
  // forward epilogue
  const float* bias;
  const bf16* out_act; const float* out_z; const bf16* out_zlow;    // null: not asked for (written through their tensor maps)
  uint32_t* relubits; int64_t w32;
  // forward epilogue that also fills the next layer's store (index part already in place)
  bf16* st_values; const uint32_t* st_keepbits; const uint32_t* st_offsets; int64_t st_capacity; int32_t st_ncb; float st_scale;
  // input-grad epilogue
  const uint32_t* relubits_prev; const bf16* z_prev; int64_t ld_zprev;
  const bf16* dz; int64_t ld_dz; float* db;    // db (optional): also the column sums of dZ
  // dW epilogue
  float* out_dw; int64_t ld_dw; int64_t dw_rows; const uint32_t* row_idx; float* partial; int64_t partial_rows;
  int32_t* dev_status;
  uint64_t wait_limit_ns;    // every device-side wait of the launch gives up after this long
  bool beside;               // forward, input gradient: runs beside the kernel ahead, and waits for its end at its own end
};

// ---- PTX wrappers ---------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) { asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory"); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
// 16 lanes x 32 columns: register 4 i + e holds lane (thread / 4) + 8 (e / 2), column 8 i + 2 (thread % 4) + e % 2.
__device__ __forceinline__ void tmem_ld16x32(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// the same where other work lies between the load and the wait: naming the registers keeps their uses behind it
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])::"memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle.  K-major: rows of 64 elements (128 B), eight
// rows form a 1024 B swizzle atom, SBO = 1024 B between atoms along M/N.  MN-major: rows of 64
// M/N elements (one per K index), SBO = 1024 B between groups of eight K rows, LBO = distance to
// the next 64 M/N elements.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) |
         ((uint64_t)(sbo_bytes >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// ---- work decomposition ---------------------------------------------------------------------------
struct Unit {
  int64_t m0, n0;
  int32_t kb0, kb1;    // K blocks [kb0, kb1)
  int32_t split;
};

// 32-bit arithmetic: a matrix that fits the device has far fewer than 2^31 tiles, and a unit's place costs half a dozen
// divisions, which nothing overlaps at the start of a launch (64-bit ones: 0.5 us before the first load).
struct Schedule {
  int64_t M;
  uint32_t m_tiles, n_tiles, ntiles, units;
  int32_t kblocks, splits, bm, bn;
  __device__ Schedule(int64_t M_, int64_t N_, int64_t K_, int32_t splits_, int32_t bm_ = BM, int32_t bn_ = BN) {
    M = M_;
    bm = bm_;
    bn = bn_;
    m_tiles = ((uint32_t)M + bm - 1) / bm;
    n_tiles = ((uint32_t)N_ + bn - 1) / bn;
    ntiles = m_tiles * n_tiles;
    kblocks = (int32_t)(((uint32_t)K_ + BK - 1) / BK);
    splits = splits_;
    units = ntiles * splits;
  }
  // split-major order: CTAs of one wave work on the same K range, so operand panels shared by
  // tiles of a row or column of the grid are read from L2 at about the same time.
  __device__ Unit unit(uint32_t u) const {
    Unit w;
    const uint32_t s = splits > 1 ? u / ntiles : 0, t = u - s * ntiles;
    const uint32_t per_group = kRasterGroup * n_tiles;
    const uint32_t g = t / per_group, r = t - g * per_group;
    const uint32_t first_m = g * kRasterGroup;
    const uint32_t gm = min((uint32_t)kRasterGroup, m_tiles - first_m), col = r / gm;
    w.m0 = (int64_t)(first_m + r - col * gm) * bm;
    w.n0 = (int64_t)col * bn;
    w.split = (int32_t)s;
    w.kb0 = splits > 1 ? (int32_t)(s * (uint32_t)kblocks / (uint32_t)splits) : 0;
    w.kb1 = splits > 1 ? (int32_t)((s + 1) * (uint32_t)kblocks / (uint32_t)splits) : kblocks;
    return w;
  }
};

// ---- epilogue of the forward pass and the input gradient ----------------------------------------------
// A thread holds one accumulator row (32 columns of it at a time).  Storing from there would touch 32 lines of the output
// per instruction for 16 bytes each, so every warp passes its chunk of 32 rows x 32 columns on through shared memory: a row
// writes its 64 bytes (bf16) or 128 (float32), 16-byte units swizzled the way the tensor map says so that eight rows take
// eight bank groups, and one TMA store takes the chunk away.  Rows and columns past the matrix are cut off by the tensor map.
// What the epilogue reads (the next store's index, ReLU bits, z of the GELU derivative) is on its way before the
// accumulators are waited for.
constexpr int kChunkBytes = 32 * 64;             // 32 rows x 32 bf16 columns
constexpr int kRingBytes = 32 * kChunkBytes;     // chunk buffers of all epilogue warps: four each of eight, two each of sixteen
constexpr int kFillBuffers = 8;                  // four lane quarters, two tiles of 128 columns
constexpr int kBiasBytes = 8 * 128 * 4;          // every warp's columns of the bias
constexpr int kSumBytes = 2 * 8 * 16 * 4;        // every warp's sums of a group of columns (bias gradient), twice
// What an epilogue takes of the shared memory; the ring of operand stages gets the rest.
constexpr int fill_bytes(int epi) { return epi >= kFwdFill && epi < kDx ? kFillBuffers * kFillBytes : 0; }
constexpr int epi_bytes(int epi) { return epi == kDwT ? 0 : kRingBytes + (is_dx(epi) ? kSumBytes : fill_bytes(epi) + kBiasBytes); }

__device__ __forceinline__ uint32_t chunk16_addr(uint32_t base, int row, int unit) { return base + row * 64 + ((unit ^ ((row >> 1) & 3)) << 4); }
__device__ __forceinline__ uint32_t chunk32_addr(uint32_t base, int row, int unit) { return base + row * 128 + ((unit ^ (row & 7)) << 4); }
__device__ __forceinline__ void st_shared16(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint4 ld_shared16(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// all but the newest `N` stores of this thread have read their shared memory
template <int N> __device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void tma_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h2);
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Where a row's activations go in the next layer's store: the part of its index (in place before the launch) that
// belongs to one row and one tile of 128 columns.
struct StoreRow {
  uint4 bits;                // the row's four keep-bit words of the tile
  uint32_t pos;              // where its first kept entry of the tile goes
  uint32_t seg, end;         // warp: kept entries of its 32 rows go to seg .. end
  bool staged;               // warp: they are collected in shared memory and copied out in 16-byte pieces, by the warps of the tile
  __device__ __forceinline__ void load(const TcParams& p, int64_t m, int64_t n, bool row_ok, bool whole_tile) {
    bits = make_uint4(0u, 0u, 0u, 0u);
    pos = end = 0u;
    if (row_ok) {
      const int64_t tile = (m >> 6) * p.st_ncb + (n >> 7);
      const uint32_t* tw = p.st_keepbits + tile * kTileWords;
      bits = *reinterpret_cast<const uint4*>(tw + (int)(m & 63) * 4);
      pos = p.st_offsets[tile] + reinterpret_cast<const unsigned short*>(tw + kBitWords)[(int)(m & 63)];
      end = pos + __popc(bits.x) + __popc(bits.y) + __popc(bits.z) + __popc(bits.w);
    }
    // the 32 rows of a warp lie in one tile, one after the other, so their kept entries are neighbours
    seg = __shfl_sync(0xffffffffu, pos, 0);
    const bool in_order = __all_sync(0xffffffffu, !row_ok || row_in_order(seg, pos, end));
    const bool fits = __all_sync(0xffffffffu, !row_ok || row_fits_stage(seg, pos, end));
    if (!in_order) raise_status(p.dev_status, RAD_DEV_EINTERNAL);      // not this store's index: entry by entry, inside `values`
    end = __reduce_max_sync(0xffffffffu, end);
    staged = whole_tile && ((uintptr_t)p.st_values & 15) == 0 && end > seg && fits;
  }
};

// This row's 32 activations (ab: rounded, two to a word) are keep-bit word `wq` of the next layer's store (Sec. 4.2: the
// layer input is what is sampled), whose index part (drawn from the key alone) is in place: the kept ones go, scaled and
// rounded, to consecutive places: into the warp's piece of shared memory at `fill`, or, where that is not used, straight to
// the store.  `buf`: the chunk buffer that holds the activations.
__device__ __forceinline__ void place_kept(const TcParams& p, const uint32_t (&ab)[16], const StoreRow& sr, int wq, uint32_t fill,
                                           uint32_t buf, int lane) {
  uint32_t word = wq == 0 ? sr.bits.x : wq == 1 ? sr.bits.y : wq == 2 ? sr.bits.z : sr.bits.w;
  uint32_t pos = sr.pos;
  if (wq > 0) pos += __popc(sr.bits.x);
  if (wq > 1) pos += __popc(sr.bits.y);
  if (wq > 2) pos += __popc(sr.bits.z);
  if (sr.staged) {
    // predicated stores, no branches: few lanes keep the same column
    uint32_t at = fill + 2u * (pos - (sr.seg & ~7u));
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
      const uint32_t a = ab[j >> 1], v = pack_bf16(__fmul_rn(bf16_lo(a), p.st_scale), __fmul_rn(bf16_hi(a), p.st_scale));
#pragma unroll
      for (int e = 0; e < 2; ++e)
        asm volatile("{\n\t.reg .pred k;\n\t.reg .b32 t;\n\tand.b32 t, %2, %3;\n\tsetp.ne.u32 k, t, 0;\n\t@k st.shared.b16 [%0], %1;\n\t"
                     "@k add.u32 %0, %0, 2;\n\t}"
                     : "+r"(at) : "h"((unsigned short)(e ? v >> 16 : v & 0xffffu)), "r"(word), "r"(1u << (j + e)) : "memory");
    }
  } else {
    const uint32_t row = buf + lane * 64;              // 16-byte unit u of the row lies at u ^ ((lane >> 1) & 3)
    const uint32_t swz = (uint32_t)((lane >> 1) & 3) << 4;
#pragma unroll 1
    while (word != 0) {
      const uint32_t c = (uint32_t)__ffs((int)word) - 1u;
      word &= word - 1u;
      unsigned short h;
      asm volatile("ld.shared.b16 %0, [%1];" : "=h"(h) : "r"(row + ((c << 1) ^ swz)) : "memory");
      const float v = __fmul_rn(__uint_as_float((uint32_t)h << 16), p.st_scale);
      if ((int64_t)pos < p.st_capacity) p.st_values[pos] = __float2bfloat16_rn(v);
      ++pos;
    }
  }
}
// The staged entries to their places, 16 bytes at a time where all eight belong to the rows, by `threads` threads.
__device__ __forceinline__ void copy_kept(const TcParams& p, const StoreRow& sr, uint32_t fill, int thread, int threads) {
  const uint32_t base = sr.seg & ~7u, end = (uint32_t)min((int64_t)sr.end, p.st_capacity);
  for (uint32_t q = base + 8u * thread; q < end; q += 8u * threads) {
    const uint4 v = ld_shared16(fill + 2u * (q - base));
    if (q >= sr.seg && q + 8u <= end) {
      *reinterpret_cast<uint4*>(p.st_values + q) = v;
    } else {
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (q + e >= sr.seg && q + e < end)
          reinterpret_cast<unsigned short*>(p.st_values)[q + e] = (unsigned short)((e & 1) ? w[e >> 1] >> 16 : w[e >> 1] & 0xffffu);
    }
  }
}
// zeros between the last value of the tile that starts with this row and its padded end
__device__ __forceinline__ void pad_store_tile(const TcParams& p, int64_t m, int64_t n) {
  const int64_t tile = (m >> 6) * p.st_ncb + (n >> 7);
  const uint32_t* tw = p.st_keepbits + tile * kTileWords;
  const uint4 last = *reinterpret_cast<const uint4*>(tw + 63 * 4);
  const uint32_t exact = reinterpret_cast<const unsigned short*>(tw + kBitWords)[63] + __popc(last.x) + __popc(last.y) +
                         __popc(last.z) + __popc(last.w);
  // 64 bits: places past 2^32 are no places of the buffer's beginning
  const uint64_t end = min((uint64_t)p.st_offsets[tile + 1], (uint64_t)p.st_capacity);
  for (uint64_t q = (uint64_t)p.st_offsets[tile] + exact; q < end; ++q) p.st_values[q] = __float2bfloat16_rn(0.0f);
}

// the ring's slot of a chunk: one, or the first of two
template <int kSlots>
__device__ __forceinline__ int chunk_slot(int turn, bool both) { return both ? turn % (kSlots / 2) * 2 : turn % kSlots; }

// One chunk of the forward pass: r holds the 32 float32 accumulators of row m, columns n .. n + 31 (as bit patterns);
// y0 is the warp's first row.  `turn` counts the warp's chunks, `stage` is its ring of kSlots chunk buffers.  Returns the chunk's ReLU bits.  The activation is a template
// parameter: what is not used is not there to be jumped over, which cost 4 us a tile of 128 x 256 (instruction fetch).
template <int ACT, int kSlots>
__device__ __forceinline__ uint32_t forward_chunk(const TcParams& p, const CUtensorMap* tm_act, const CUtensorMap* tm_zlow,
                                                  const CUtensorMap* tm_z, const uint32_t (&r)[32], int y0, int n, int lane,
                                                  uint32_t stage, uint32_t bias, int turn, uint32_t (&ab)[16]) {
  const int nvalid = min(32, (int)p.N - n);      // multiple of 8
  float v[32];
  if (p.bias != nullptr) {
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
      const uint4 b4 = ld_shared16(bias + 4 * j);
      v[j] = __uint_as_float(r[j]) + __uint_as_float(b4.x); v[j + 1] = __uint_as_float(r[j + 1]) + __uint_as_float(b4.y);
      v[j + 2] = __uint_as_float(r[j + 2]) + __uint_as_float(b4.z); v[j + 3] = __uint_as_float(r[j + 3]) + __uint_as_float(b4.w);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
  }
  const bool z_only = p.out_act == nullptr && p.out_zlow == nullptr;
  if (p.out_z != nullptr) {
    // buffers of 4 KB; where 16-bit results follow they share the ring
    const uint32_t buf = z_only ? stage + turn % (kSlots / 2) * 2 * kChunkBytes : stage;
    if (elect_one()) {
      if (z_only) tma_store_wait_read<kSlots / 2 - 1>();
      else tma_store_wait_read<0>();
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; j += 4)
      st_shared16(chunk32_addr(buf, lane, j >> 2), __float_as_uint(v[j]), __float_as_uint(v[j + 1]), __float_as_uint(v[j + 2]),
                  __float_as_uint(v[j + 3]));
    fence_proxy_async();
    __syncwarp();
    if (elect_one()) {
      tma_store_2d(tm_z, n, y0, buf);
      tma_store_commit();
    }
    if (z_only) return 0u;
  }
  uint32_t zl[16], bits = 0;
  if (p.out_zlow != nullptr) {
#pragma unroll
    for (int j = 0; j < 32; j += 2) zl[j >> 1] = pack_bf16(v[j], v[j + 1]);
  }
  if (p.out_act != nullptr) {
    if (ACT == RAD_ACT_GELU) {
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = gelu_f(v[j]);
    } else if (ACT == RAD_ACT_RELU) {
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = fmaxf(v[j], 0.0f);
    }
#pragma unroll
    for (int j = 0; j < 32; j += 2) ab[j >> 1] = pack_bf16(v[j], v[j + 1]);
    if (p.relubits != nullptr) {
      // The bit is taken from the rounded activation, the tensor the backward sees.  A comparison gives a mask for the two
      // halves of a word; pair i leaves its column 2 i in bit i and 2 i + 1 in bit 16 + i, and the halves are interleaved last.
      const __nv_bfloat162 zero = __floats2bfloat162_rn(0.0f, 0.0f);
#pragma unroll
      for (int i = 0; i < 16; ++i)
        bits |= __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&ab[i]), zero) & (0x00010001u << i);
      uint32_t t = (bits ^ (bits >> 8)) & 0x0000ff00u;
      bits ^= t ^ (t << 8);
      t = (bits ^ (bits >> 4)) & 0x00f000f0u;
      bits ^= t ^ (t << 4);
      t = (bits ^ (bits >> 2)) & 0x0c0c0c0cu;
      bits ^= t ^ (t << 2);
      t = (bits ^ (bits >> 1)) & 0x22222222u;
      bits ^= t ^ (t << 1);
    }
  }
  // one output takes a buffer of the ring a chunk, two take a pair of them
  const bool both = p.out_zlow != nullptr && p.out_act != nullptr;
  if (turn >= kSlots / 2 || p.out_z != nullptr) {
    if (elect_one()) {
      if (p.out_z != nullptr) tma_store_wait_read<0>();
      else if (both) tma_store_wait_read<kSlots / 2 - 1>();
      else tma_store_wait_read<kSlots - 1>();
    }
    __syncwarp();
  }
  const uint32_t first = stage + chunk_slot<kSlots>(turn, both) * kChunkBytes, second = first + kChunkBytes;
  if (p.out_act != nullptr) {
#pragma unroll
    for (int u = 0; u < 4; ++u) st_shared16(chunk16_addr(first, lane, u), ab[4 * u], ab[4 * u + 1], ab[4 * u + 2], ab[4 * u + 3]);
  }
  if (p.out_zlow != nullptr) {
    const uint32_t to = both ? second : first;
#pragma unroll
    for (int u = 0; u < 4; ++u) st_shared16(chunk16_addr(to, lane, u), zl[4 * u], zl[4 * u + 1], zl[4 * u + 2], zl[4 * u + 3]);
  }
  fence_proxy_async();
  __syncwarp();
  if (elect_one()) {
    if (p.out_act != nullptr) tma_store_2d(tm_act, n, y0, first);
    if (p.out_zlow != nullptr) tma_store_2d(tm_zlow, n, y0, both ? second : first);
    tma_store_commit();
  }
  // columns past the layer's width are not activations
  return nvalid < 32 ? bits & ((1u << nvalid) - 1u) : bits;
}

// z of the GELU derivative for a warp's chunk (32 rows from y0, 32 columns from n) into shared memory, four lanes to a row.
__device__ __forceinline__ void prefetch_z(const TcParams& p, int64_t y0, int64_t n, int lane, uint32_t buf) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = 8 * i + (lane >> 2), unit = lane & 3;
    if (y0 + row < p.M && n + 8 * unit < p.N)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                   ::"r"(chunk16_addr(buf, row, unit)), "l"(p.z_prev + (y0 + row) * p.ld_zprev + n + 8 * unit) : "memory");
  }
}
// One chunk of the input gradient: times the derivative of the activation before (ReLU bits, or GELU' of the z that lies in
// `buf`), rounded, out through the same buffer.  GELU' is the function of the CUDA-core route, so that a net's gradients do not
// depend on the route a shape takes.  Its erff and exponential are what bounds a GELU net's input gradient of few inputs.  They
// are made for eight columns a turn: with the code of 32 in one piece, which every warp fetches anew for every chunk, 16384 x
// 2048 x 1024 took 95 us instead of 79, 16384 x 4096 x 64 166 instead of 128 (sixteen warps: 123 for the latter, but more where
// the MMAs bound: 4096 x 2048 x 2048 32.7 against 30.9).
template <bool kGelu>
__device__ __forceinline__ void dx_chunk(const CUtensorMap* tm_dx, uint32_t taddr, int y0, int n, int lane, uint32_t bits, uint32_t buf) {
  if (kGelu) {
#pragma unroll 1
    for (int u = 0; u < 4; ++u) {
      uint32_t r[8];
      tmem_ld8(taddr + 8 * u, r);
      const uint32_t at = chunk16_addr(buf, lane, u);
      const uint4 zq = ld_shared16(at);
      const uint32_t zw[4] = {zq.x, zq.y, zq.z, zq.w};
      float g[8];
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        g[e] = gelu_grad_f(bf16_lo(zw[e >> 1]));
        g[e + 1] = gelu_grad_f(bf16_hi(zw[e >> 1]));
      }
      tmem_ld_wait(r);
#pragma unroll
      for (int e = 0; e < 8; ++e) g[e] *= ((bits >> e) & 1u) ? __uint_as_float(r[e]) : 0.0f;
      st_shared16(at, pack_bf16(g[0], g[1]), pack_bf16(g[2], g[3]), pack_bf16(g[4], g[5]), pack_bf16(g[6], g[7]));
      bits >>= 8;
    }
  } else {
    uint32_t r[32];
    tmem_ld32(taddr, r);
    tmem_ld_wait();
    float g[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) g[j] = ((bits >> j) & 1u) ? __uint_as_float(r[j]) : 0.0f;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      st_shared16(chunk16_addr(buf, lane, u), pack_bf16(g[8 * u], g[8 * u + 1]), pack_bf16(g[8 * u + 2], g[8 * u + 3]),
                  pack_bf16(g[8 * u + 4], g[8 * u + 5]), pack_bf16(g[8 * u + 6], g[8 * u + 7]));
  }
  fence_proxy_async();
  __syncwarp();
  if (elect_one()) {
    tma_store_2d(tm_dx, n, y0, buf);
    tma_store_commit();
  }
}

// Different-sample dW: 32 accumulator rows (from row `m0`, tensor-memory address `taddr`) x 32 columns by one warp.
// With a row per thread every 16-byte store of a warp touches 32 lines, one look-up each: 8 us for a CTA's 128 x 512
// tile, whatever the number of warps.  Here the accumulators come in the layout of matrix fragments and neighbouring
// threads exchange column pairs, so that a store covers 64 bytes of eight rows.
__device__ __forceinline__ void epilogue_dw(const TcParams& p, uint32_t taddr, int64_t m0, int64_t n, int32_t split, int lane) {
  const int nvalid = (int)min((int64_t)32, p.N - n);      // multiple of 8
  uint32_t r[2][16];
  tmem_ld16x32(taddr, r[0]);
  tmem_ld16x32(taddr + (16u << 16), r[1]);
  tmem_ld_wait();
  const bool odd = (lane & 1) != 0;
#pragma unroll
  for (int h = 0; h < 4; ++h) {                            // rows 8 h + lane / 4
    const int64_t m = m0 + 8 * h + (lane >> 2);
    float* dst = p.splits > 1 ? p.partial + ((int64_t)split * p.partial_rows + m) * p.N + n : p.out_dw + m * p.ld_dw + n;
#pragma unroll
    for (int i = 0; i < 4; i += 2) {                       // column blocks i (even threads keep it) and i + 1 (odd threads)
      const uint32_t* a = &r[h >> 1][4 * i + 2 * (h & 1)];
      const uint32_t* b = a + 4;
      const uint32_t t0 = __shfl_xor_sync(0xffffffffu, odd ? a[0] : b[0], 1);
      const uint32_t t1 = __shfl_xor_sync(0xffffffffu, odd ? a[1] : b[1], 1);
      const float4 v = odd ? make_float4(__uint_as_float(t0), __uint_as_float(t1), __uint_as_float(b[0]), __uint_as_float(b[1]))
                           : make_float4(__uint_as_float(a[0]), __uint_as_float(a[1]), __uint_as_float(t0), __uint_as_float(t1));
      const int col = 8 * (i + (lane & 1)) + 4 * ((lane >> 1) & 1);
      if (m < p.M && col < nvalid) *reinterpret_cast<float4*>(dst + col) = v;
    }
  }
}

// Same-sample dW, transposed tile: the accumulator row is output column h of dW, the accumulator column is
// kept column j; r holds dW[idx[n + jj], h] for jj < 32.  For a fixed jj the 32 lanes of a warp write 32
// consecutive floats of one row of dW (or of the split's partial block, row n + jj).
__device__ __forceinline__ void epilogue_chunk_dwt(const TcParams& p, const uint32_t (&r)[32], int64_t h, int64_t n,
                                                   int nvalid, bool row_ok, int32_t split) {
  if (!row_ok) return;
  if (p.splits > 1) {
    float* dst = p.partial + ((int64_t)split * p.partial_rows + n) * p.M + h;
#pragma unroll
    for (int jj = 0; jj < 32; ++jj)
      if (jj < nvalid) dst[(int64_t)jj * p.M] = __uint_as_float(r[jj]);
  } else {
#pragma unroll
    for (int j0 = 0; j0 < 32; j0 += 8) {          // the rows of eight columns are read before the first of their stores
      uint32_t row[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (j0 + e < nvalid) row[e] = p.row_idx[n + j0 + e];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (j0 + e < nvalid) {
          if (row[e] < p.dw_rows) p.out_dw[row[e] * p.ld_dw + h] = __uint_as_float(r[j0 + e]);
          else raise_status(p.dev_status, RAD_DEV_EINTERNAL);
        }
      }
    }
  }
}

// ---- bias gradient beside the input gradient ------------------------------------------------------------
// The epilogue warps have nothing to do while the MMAs of a tile run, so they add up the columns of dZ meanwhile, a share
// of the work per tile: a CTA takes groups of 16 columns (8 where that gives every CTA a group: 32 bytes of a row are a
// sector), a thread 16 bytes of every (256 >> shift)-th row, eight loads in flight.  As a launch of its own this took 4 to 9
// us behind every input gradient of a net of ordinary size, and 0.2 ms at 65536 x 8192.
// Sums of eight rows as a tree, then one after the other, then over lanes and warps.
struct ColumnSums {
  float acc[8];
  uint32_t group, step, turn;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
  }
};
constexpr int kSumThreads = 256, kSumLoads = 8;
__host__ __device__ constexpr int sum_shift(int64_t columns, int64_t ctas) { return columns > 8 * ctas ? 1 : 0; }   // 16-byte loads a row: 1 or 2
__device__ __forceinline__ void add_bf16x8(const uint4& q, float (&v)[8]) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] += bf16_lo(w[i]);
    v[2 * i + 1] += bf16_hi(w[i]);
  }
}
// One step: kSumLoads rows a thread.
__device__ __forceinline__ void column_sums_step(const TcParams& p, ColumnSums& cs, int shift, int thread) {
  const int64_t col = ((int64_t)cs.group << shift) * 8 + 8 * (thread & ((1 << shift) - 1));
  const uint32_t lanes = kSumThreads >> shift;
  const int64_t row0 = (int64_t)cs.step * lanes * kSumLoads + (thread >> shift);
  uint4 q[kSumLoads];
#pragma unroll
  for (int j = 0; j < kSumLoads; ++j) {
    const int64_t row = row0 + (int64_t)j * lanes;
    q[j] = make_uint4(0u, 0u, 0u, 0u);
    if (row < p.M && col < p.K) q[j] = *reinterpret_cast<const uint4*>(p.dz + row * p.ld_dz + col);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float v[8];
    const uint32_t w[4] = {q[4 * h].x, q[4 * h].y, q[4 * h].z, q[4 * h].w};
    float u[8];
    const uint32_t x[4] = {q[4 * h + 2].x, q[4 * h + 2].y, q[4 * h + 2].z, q[4 * h + 2].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[2 * i] = bf16_lo(w[i]);
      v[2 * i + 1] = bf16_hi(w[i]);
      u[2 * i] = bf16_lo(x[i]);
      u[2 * i + 1] = bf16_hi(x[i]);
    }
    add_bf16x8(q[4 * h + 1], v);
    add_bf16x8(q[4 * h + 3], u);
#pragma unroll
    for (int i = 0; i < 8; ++i) cs.acc[i] += v[i] + u[i];
  }
}
// A warp's sums of the group it has gone through, into `red` (16 columns).
__device__ __forceinline__ void column_sums_warp(ColumnSums& cs, int shift, int lane, float* red) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (o < (1 << shift)) continue;
#pragma unroll
    for (int i = 0; i < 8; ++i) cs.acc[i] += __shfl_xor_sync(0xffffffffu, cs.acc[i], o);
  }
  if (lane < (1 << shift)) {
#pragma unroll
    for (int i = 0; i < 8; ++i) red[8 * lane + i] = cs.acc[i];
  }
  cs.clear();
}

// ---- shared memory layout -------------------------------------------------------------------------
constexpr int kIndexBytes = kTileWords * 4;   // keep bits + row offsets of one store tile (1152 B)
constexpr int kFirstExpanderWarp = 7;        // warp 6 feeds the compressed ring
// ---- expansion of one keep-bit word into the A_hat tile -------------------------------------------
// sA: the stage's A tile (four 8 KB blocks of 64 columns, 128-byte rows per K index, 128-byte
// swizzle); sC: keep bits, row offsets and packed values of store tile h of this K block; the thread
// owns row r, columns 32 wq .. 32 wq + 31 of that store tile.  limit: staged values per tile.
__device__ __forceinline__ void expand_word(uint8_t* sA, const uint8_t* sC, int h, int r, int wq, uint32_t limit) {
  const uint32_t* bits = reinterpret_cast<const uint32_t*>(sC);
  const unsigned short* rowoff = reinterpret_cast<const unsigned short*>(sC + kBitWords * 4);
  const unsigned short* vals = reinterpret_cast<const unsigned short*>(sC + kIndexBytes);
  const uint4 rowbits = *reinterpret_cast<const uint4*>(bits + r * 4);
  const uint32_t word = wq == 0 ? rowbits.x : wq == 1 ? rowbits.y : wq == 2 ? rowbits.z : rowbits.w;
  uint32_t pos = rowoff[r];
  if (wq > 0) pos += __popc(rowbits.x);
  if (wq > 1) pos += __popc(rowbits.y);
  if (wq > 2) pos += __popc(rowbits.z);
  uint8_t* rowp = sA + h * 16384 + (wq >> 1) * 8192 + r * 128;
  const int j0 = (wq & 1) * 4;
  const uint32_t cnt = __popc(word);
  // one path per warp: the dense form is right for any word
  if (__all_sync(0xffffffffu, cnt + (pos & 3u) <= 12u && cnt <= 10u)) {
    // sparse word: zero this thread's 32 columns, then drop the kept values in place.  The
    // values are consecutive from `pos`: three aligned 8-byte loads cover them (a word whose
    // values would pass the end of the staged tile places nothing: the producer has flagged it).
    // Byte address of column c of this word in the swizzled row: base ^ (c << 1), because the
    // 16-byte chunk index (j0 + (c >> 3)) ^ (r & 7) equals (c >> 3) ^ (j0 ^ (r & 7)) for j0 in {0, 4}
    // and rows are 128-byte aligned.
    const uint32_t base = smem_u32(rowp) ^ ((uint32_t)(j0 ^ (r & 7)) << 4);
#pragma unroll
    for (int jj = 0; jj < 4; ++jj)
      asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(base ^ (uint32_t)(jj << 4)), "r"(0u) : "memory");
    const uint32_t rest = (pos + cnt <= limit) ? word : 0u;
    const uint32_t e0 = pos & 3u;
    const uint2* win = reinterpret_cast<const uint2*>(vals + (min(pos, limit) & ~3u));   // stays inside the ring
    const uint2 q0 = win[0], q1 = win[1];
    uint2 q2 = make_uint2(0u, 0u);
    if (e0 + cnt > 8u) q2 = win[2];
    // bring the first kept value to bit 0 of s0: drop whole words, then a half word
    const bool drop = (e0 & 2u) != 0u;
    const uint32_t w0 = drop ? q0.y : q0.x, w1 = drop ? q1.x : q0.y, w2 = drop ? q1.y : q1.x;
    const uint32_t w3 = drop ? q2.x : q1.y, w4 = drop ? q2.y : q2.x, w5 = drop ? 0u : q2.y;
    const uint32_t sh = (e0 & 1u) << 4;
    const uint32_t sv[5] = {__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh), __funnelshift_r(w2, w3, sh),
                            __funnelshift_r(w3, w4, sh), __funnelshift_r(w4, w5, sh)};
    // every lane runs the warp's longest word; a lane that has run out stores nothing.  The word is
    // bit-reversed so that the next kept column is a leading-zero count away.
    const uint32_t steps = __reduce_max_sync(0xffffffffu, rest != 0u ? cnt : 0u);
    uint32_t rw = __brev(rest);
#pragma unroll
    for (int i = 0; i < 10; ++i) {
      if ((uint32_t)i >= steps) break;                  // warp-uniform
      const uint32_t c = (uint32_t)__clz((int)rw);      // 32 once the word is used up
      const uint32_t v = sv[i >> 1] >> (16 * (i & 1));
      asm volatile("{\n\t.reg .pred k;\n\tsetp.ne.u32 k, %2, 0;\n\t@k st.shared.b16 [%0], %1;\n\t}"
                   ::"r"(base ^ (c << 1)), "h"((unsigned short)v), "r"(rw) : "memory");
      rw &= ~(0x80000000u >> (c & 31u));
    }
  } else {
    // dense word: every column's value position follows from a popcount of the bits below
    // it, so the 32 loads are independent; each 16-byte chunk is written once
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      uint32_t pk[4];
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const int b0 = jj * 8 + e;
        const uint32_t p0 = pos + __popc(word & ((1u << b0) - 1u));
        const uint32_t p1 = pos + __popc(word & ((2u << b0) - 1u));
        const uint32_t v0 = ((word >> b0) & 1u) && p0 < limit ? vals[p0] : 0u;
        const uint32_t v1 = ((word >> (b0 + 1)) & 1u) && p1 < limit ? vals[p1] : 0u;
        pk[e >> 1] = v0 | (v1 << 16);
      }
      *reinterpret_cast<uint4*>(rowp + (((j0 + jj) ^ (r & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
  }
}

// ---- two-CTA engine (dense operands) -----------------------------------------------------------------
// A cluster of two CTAs (one SM pair) owns an output tile of 256 rows and 256, 128 or 64 columns.  Each CTA stages 128 rows of
// the A tile and 128 rows (N) of the B tile per K block and keeps 128 accumulator rows in its own
// tensor memory; one thread of the even CTA issues tcgen05.mma.cta_group::2, which reads both
// CTAs' shared memory.  Against the one-CTA tile this halves the operand bytes each SM's shared
// memory has to deliver per MMA, and a 128 x 256 accumulator takes 256 tensor-memory columns, so
// two of them alternate: the epilogue of one tile runs under the MMAs of the next.
// Barriers: full[s] (even CTA; its producer arrives once with the byte count of both CTAs, and
// both CTAs' TMA complete on it: the odd CTA reloads a stage only after the commit that follows the
// even CTA's wait on the previous phase, so its bytes never reach an older phase), empty[s] and tmem_full[b] (one per CTA, signalled by the MMA thread's commit to
// both CTAs), tmem_empty[b] (even CTA; every epilogue warp of the pair arrives).
// A stage is 16 KB of A and as much of B as the tile is wide (MN-major: in boxes of 64 columns), and as many stages as there is
// room for are in flight: narrow tiles of long contractions wait for memory and not for the tensor core.  Us with four stages
// of 32 KB / so: 32768 x 4096 to 64 columns, input gradient 61.6 / 53.9, same-sample dW, which has no epilogue buffers and
// whose width only the device knows, 51.6 / 46.9 (16384 x 4096 x 1024: 39.5 / 33.6); forward: see dense_tile_width.
constexpr int kStage2ABytes = 128 * BK * 2;
constexpr int kStages2 = 6;
constexpr int stage2_bytes(int bkind, int bn) { return kStage2ABytes + (bkind == kBK_ ? bn / 2 * BK * 2 : (bn / 2 + 63) / 64 * 8192); }
// Epilogue warps, eight or sixteen.  Sixteen for a forward pass of up to kWideEpilogueK inputs that places the next layer's store
// and for a GELU of up to kWideGeluK inputs: more warps hide the latencies of erff and of the stores (a tile of 256 x 256 in us,
// eight / sixteen: GELU 7.3 / 6.3, with pre-activations and store 10.3 / 9.9, ReLU with store 5.7 / 5.7); with more inputs the
// MMAs of a tile outlast the epilogue of the one before, and where a GELU without a store also writes the pre-activations of
// many tiles eight were faster (16384 x 512 x 4096 186 / 196).
constexpr int64_t kWideEpilogueK = 2048, kWideGeluK = 1024, kWideGeluWaves = 4;
constexpr int threads2(int epi_warps) { return 32 * (2 + epi_warps); }
// A quarter of an SM holds three of ten warps, or five of eighteen, and one of a small kernel of another stream has to fit
// beside them (with 168 registers a thread, of ten warps, such a kernel waited for the end of the launch;
// tests/test_gpu_streams.py).
constexpr int register_bound2(int epi_warps) { return epi_warps == 8 ? 144 : 96; }

struct SmemCtl2 {
  uint64_t full[kStages2], empty[kStages2], tmem_full[2], tmem_empty[2], group[kFillBuffers];
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ uint32_t map_to_cta(uint32_t saddr, uint32_t rank) {   // shared::cluster address
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Arrival on a barrier of either CTA of the pair (default semantics, as for a local arrival: what
// the waiter goes on to touch is ordered by tcgen05 or proxy fences issued before the arrival; a
// cluster-scope release here would drain the SM's outstanding stores every time).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t caddr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(caddr) : "memory");
}
// What a bounded wait of the pair needs: this CTA's abort flag, the peer's (shared::cluster address) and
// the time limit of the launch (a kernel argument; rad_set_wait_limit_ns).
struct PairWait {
  volatile int* abort_flag;
  uint32_t peer_abort;
  uint64_t limit_ns;
};
// Bounded wait of the pair: on expiry both CTAs' abort flags are raised.  sleep_ns > 0: a long wait
// off the critical path (an epilogue warp waiting for a whole tile) leaves the issue slots to others.
__device__ __forceinline__ bool mbar_wait2(uint32_t bar, uint32_t parity, const PairWait& wc, uint32_t sleep_ns = 0) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 32; ++i) {
      if (mbar_try_wait(bar, parity)) return true;
      if (sleep_ns != 0) __nanosleep(sleep_ns);
    }
    if (*wc.abort_flag != 0) return false;
    if (global_timer_ns() - t0 > wc.limit_ns) {
      *wc.abort_flag = 1;
      asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(wc.peer_abort), "r"(1u) : "memory");
      return false;
    }
  }
}
// Several warps meet on a barrier that one lane of each arrives at and waits for (a bounded wait like the others): what any of
// their threads wrote to shared memory before is seen by all of them after it.  The waiting lane has seen the others' writes,
// and a warp barrier, which a shuffle is not, hands that on to its warp.
__device__ __forceinline__ bool warps_meet(uint32_t bar, uint32_t parity, const PairWait& wc, int lane) {
  __syncwarp();
  bool met = true;
  if (lane == 0) {
    mbar_arrive(bar);
    met = mbar_wait2(bar, parity, wc);
  }
  met = __shfl_sync(0xffffffffu, met ? 1 : 0, 0) != 0;
  __syncwarp();
  return met;
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t cbar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(cbar), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {   // the barrier at this offset in both CTAs
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((unsigned short)3) : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// D = f32, A = B = bf16, M = 256 over the pair, N = n (a multiple of 16, at most 256).
__host__ __device__ constexpr uint32_t make_idesc_pair(bool a_mn, bool b_mn, uint32_t n = 256u) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((n >> 3) << 17) | ((256u >> 4) << 24);
}

// The tensor maps of the outputs: tmO activation or input gradient, tmL pre-activation in bf16, tmZ float32 results.
template <int AK, int BKIND, int EPI, int kEpiWarps>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(register_bound2(kEpiWarps))
tc_gemm_pair_kernel(const TcParams p, const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmL,
                    const __grid_constant__ CUtensorMap tmZ) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int stages = p.num_stages, stage_bytes = stage2_bytes(BKIND, EPI == kDwT ? BN : p.bn);
  uint8_t* epi_smem = smem + (size_t)stages * stage_bytes;
  SmemCtl2* ctl = reinterpret_cast<SmemCtl2*>(epi_smem + epi_bytes(EPI));
  volatile int* abort_flag = &ctl->abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();         // 0: issues the MMAs; both stage operands and run epilogues
  const uint32_t peer_abort = map_to_cta(smem_u32(&ctl->abort_flag), rank ^ 1u);
  const PairWait wc = {abort_flag, peer_abort, p.wait_limit_ns};
  const uint32_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  if (tid == 0) {
    prefetch_map(&tmA);
    prefetch_map(&tmB);
    if (EPI != kDwT) prefetch_map(p.out_z != nullptr ? &tmZ : &tmO);
    for (int s = 0; s < stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&ctl->tmem_full[b]), 1);
      mbar_init(smem_u32(&ctl->tmem_empty[b]), 2 * kEpiWarps);
    }
    if (is_dx(EPI)) mbar_init(smem_u32(&ctl->group[0]), kEpiWarps);       // all of them, for the bias gradient
    if (is_forward(EPI))             // the warps that fill one store tile together: four in a tile of 32 columns each
      for (int g = 0; g < kFillBuffers; ++g) mbar_init(smem_u32(&ctl->group[g]), p.bn == 256 ? kEpiWarps / 8 : kEpiWarps / 4);
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {   // the same warp of both CTAs allocates for the pair: two 128 x 256 accumulators per CTA
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&ctl->tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_barrier();        // the peer's barriers are initialised before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  const uint32_t smem_base = smem_u32(smem);
  // so far nothing of another kernel was touched: the above runs under the tail of the kernel before, and so does the
  // division of the work, which depends on the parameters only (not for kDwT)
  if (EPI == kDwT) wait_for_previous();
  // Same-sample dW (kDwT): the tile is dW^T, M = H, N = kept columns (known on the device only).  The kept
  // columns are cut into the fewest tiles of at most 256 and the tile width bn is what one of them needs,
  // rounded up to the MMA's granule of 16: 105 kept columns cost one tile of 112, not one of 256.
  int64_t n_cols = p.N;
  int bn = p.bn;
  if (EPI == kDwT) {
    int64_t nd;
    asm volatile("ld.global.cg.s64 %0, [%1];" : "=l"(nd) : "l"(p.N_dev) : "memory");
    n_cols = nd < n_cols ? nd : n_cols;
    const int64_t nt = max((int64_t)1, (n_cols + BN - 1) / BN);
    bn = max(16, (int)(((n_cols + nt - 1) / nt + 15) / 16 * 16));
  }
  const Schedule sched(p.M, n_cols, p.K, p.splits, BM, bn);
  if (EPI != kDwT && !p.beside) wait_for_previous();
  const int boxes_b = (bn / 2 + 63) / 64;             // 64-column boxes of an MN-major B this CTA stages per K block
  const uint32_t stage_tx = 2u * (uint32_t)(kStage2ABytes + (BKIND == kBK_ ? bn / 2 * 128 : boxes_b * 8192));

  if (warp == 0) {
    // ===== TMA producer: this CTA's 128 rows of A and 128 rows (N) of B, completing on the even CTA's barrier =====
    if (elect_one()) {
      const uint32_t full0 = map_to_cta(smem_u32(&ctl->full[0]), 0u);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
        const Unit w = sched.unit(u);
        if (u + npairs >= sched.units) let_next_start();
        const int m_own = (int)w.m0 + 128 * (int)rank, n_own = (int)w.n0 + (bn / 2) * (int)rank;
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          ok = mbar_wait2(smem_u32(&ctl->empty[0]) + 8u * stage, phase ^ 1u, wc);
          if (!ok) break;
          const uint32_t sA = smem_base + stage * stage_bytes;
          const uint32_t sB = sA + kStage2ABytes;
          const uint32_t full = full0 + 8u * stage;
          const int k0 = kb * BK;
          if (rank == 0) mbar_arrive_expect_tx(smem_u32(&ctl->full[0]) + 8u * stage, stage_tx);   // both CTAs' bytes
          if (AK == kAK) {
            tma_load_2d_pair(sA, &tmA, k0, m_own, full);                         // 64 (K) x 128 rows
          } else {
#pragma unroll
            for (int c = 0; c < 2; ++c) tma_load_2d_pair(sA + c * 8192, &tmA, m_own + c * 64, k0, full);
          }
          if (BKIND == kBK_) {
            tma_load_2d_pair(sB, &tmB, k0, n_own, full);
          } else {
#pragma unroll
            for (int c = 0; c < 2; ++c)
              if (c < boxes_b) tma_load_2d_pair(sB + c * 8192, &tmB, n_own + c * 64, k0, full);
          }
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
      }
      // tail: every commit aimed at this CTA's stage barriers has landed before the CTA may leave
      for (int i = 0; i < stages && ok; ++i) {
        ok = mbar_wait2(smem_u32(&ctl->empty[0]) + 8u * stage, phase ^ 1u, wc);
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ===== MMA issuer: one thread of the even CTA drives both tensor cores =====
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = make_idesc_pair(AK != kAK, BKIND == kBMN, (uint32_t)bn);
      // descriptors of stage 0; a step of 16 K rows and a stage are additions to the address field
      const uint64_t adesc0 = AK == kAK ? make_desc(smem_base, 16, 1024) : make_desc(smem_base, 8192, 1024);
      const uint64_t bdesc0 = BKIND == kBK_ ? make_desc(smem_base + kStage2ABytes, 16, 1024)
                                            : make_desc(smem_base + kStage2ABytes, 8192, 1024);
      constexpr uint32_t a_step = (AK == kAK ? 32 : 2048) >> 4, b_step = (BKIND == kBK_ ? 32 : 2048) >> 4;
      int stage = 0, buf = 0;
      uint32_t phase = 0, buf_phases = 0;          // bit b: phase of accumulator b
      bool ok = true;
      for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
        const Unit w = sched.unit(u);
        ok = mbar_wait2(smem_u32(&ctl->tmem_empty[0]) + 8u * buf, ((buf_phases >> buf) & 1u) ^ 1u, wc);
        if (!ok) break;
        tc_fence_after();
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          ok = mbar_wait2(smem_u32(&ctl->full[0]) + 8u * stage, phase, wc);
          if (!ok) break;
          tc_fence_after();
          const uint64_t adesc = adesc0 + (uint32_t)(stage * (stage_bytes >> 4));
          const uint64_t bdesc = bdesc0 + (uint32_t)(stage * (stage_bytes >> 4));
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            tc_mma_pair(tmem_base + buf * 256, adesc + k * a_step, bdesc + k * b_step, idesc, (kb > w.kb0 || k > 0) ? 1u : 0u);
          tc_commit_pair(smem_u32(&ctl->empty[0]) + 8u * stage);           // frees the stage in both CTAs
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
        if (ok) tc_commit_pair(smem_u32(&ctl->tmem_full[0]) + 8u * buf);
        buf_phases ^= 1u << buf;
        buf ^= 1;
      }
    }
    __syncwarp();
  } else {
    // ===== epilogue: thread = one accumulator row of this CTA =====
    const int q = warp & 3;
    // the warps of a lane quarter split the tile's 32-column chunks between them
    constexpr int kPerQuarter = kEpiWarps / 4;
    const int chunks = (bn + 31) / 32, own_chunks = (chunks + kPerQuarter - 1) / kPerQuarter;
    const int c_first = ((warp - 2) >> 2) * own_chunks * 32;
    const int c_last = min(c_first + own_chunks * 32, chunks * 32);
    const uint32_t empty_bar = map_to_cta(smem_u32(&ctl->tmem_empty[0]), 0u);     // [b] is 8 bytes further
    constexpr int kSlots = 32 / kEpiWarps;
    const uint32_t stage = smem_u32(epi_smem) + (warp - 2) * kSlots * kChunkBytes;
    const uint32_t bias_row = smem_u32(epi_smem) + kRingBytes + fill_bytes(EPI) + (warp - 2) * (kBiasBytes / kEpiWarps);
    // the warps of a lane quarter whose columns make up one store tile fill one buffer and copy it out together
    const bool whole_tile = bn >= 128;
    const int group = whole_tile ? 4 / own_chunks : 1, first_tile = ((warp - 2) >> 2) / group;
    const uint32_t fill = smem_u32(epi_smem) + kRingBytes + (q + 4 * (first_tile & 1)) * kFillBytes;
    const int group_thread = lane + 32 * (((warp - 2) >> 2) % group);
    const uint32_t group_bar = smem_u32(&ctl->group[q + 4 * (first_tile & 1)]);
    uint32_t group_phase = 0;
    const auto group_sync = [&]() -> bool {
      if (group == 1) { __syncwarp(); return true; }
      const bool met = warps_meet(group_bar, group_phase, wc, lane);
      group_phase ^= 1u;
      return met;
    };
    int buf = 0, turn = 0;
    uint32_t buf_phases = 0;
    bool ok = true;
    // bias gradient: this CTA's column groups are blockIdx.x, blockIdx.x + gridDim.x, ...; `quota` steps per tile
    ColumnSums cs;
    cs.clear();
    cs.group = blockIdx.x; cs.step = 0; cs.turn = 0;
    const int et = tid - 64;                           // 0 .. 32 kEpiWarps - 1
    const int shift = sum_shift(p.K, (int64_t)gridDim.x);
    uint32_t sum_groups = 0, sum_steps = 0, quota = 0;
    if (is_dx(EPI) && p.db != nullptr) {
      const uint32_t rows = (kSumThreads >> shift) * kSumLoads, cols = 8u << shift;
      sum_groups = ((uint32_t)p.K + cols - 1) / cols;
      sum_steps = ((uint32_t)p.M + rows - 1) / rows;
      const uint32_t own_groups = cs.group < sum_groups ? (sum_groups - cs.group + gridDim.x - 1) / gridDim.x : 0;
      const uint32_t own_units = (sched.units - pair + npairs - 1) / npairs;
      quota = (own_groups * sum_steps + own_units - 1) / own_units;
    }
    if (EPI == kDwT && p.keep_cols != nullptr) {
      // Rows of dW whose column was not kept are zero (Sec. 4.3: only the sampled part of the weight matrix
      // gets a gradient).  The epilogue warps have nothing to do until the first tile's MMAs retire, so they
      // write those rows now: row d belongs to CTA d mod grid, a thread writes 16 bytes at a time.
      const int64_t h4 = p.M / 4;
      for (int64_t d = blockIdx.x; d < p.dw_rows; d += gridDim.x) {
        if ((p.keep_cols[d >> 5] >> (d & 31)) & 1u) continue;
        float4* rowp = reinterpret_cast<float4*>(p.out_dw + d * p.ld_dw);
        for (int64_t i = et; i < h4; i += 32 * kEpiWarps) rowp[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
      const Unit w = sched.unit(u);
      const int64_t m_warp = w.m0 + 128 * (int64_t)rank + q * 32, m = m_warp + lane;
      const bool row_ok = m < sched.M;
      // (sixteen warps are more than a tile of 64 columns has chunks: the last ones have nothing to do)
      const int64_t n_warp = c_first < c_last ? w.n0 + c_first : n_cols, n_tile = n_warp & ~(int64_t)127;
      // what the epilogue reads besides the accumulators comes while the MMAs run (a warp's columns lie in one store tile)
      StoreRow sr = {};
      uint32_t prev_bits[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu}, act_bits[4] = {};
      if (EPI >= kFwdFill && EPI < kDx && c_first < c_last && n_tile < n_cols) {
        sr.load(p, m, n_tile, row_ok, whole_tile);
        if (row_ok && (m & 63) == 0 && (n_warp & 127) == 0) pad_store_tile(p, m, n_warp);
      }
      if (is_forward(EPI) && p.bias != nullptr) {
        // four columns a lane; zero past the layer's width
        float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (4 * lane < 32 * own_chunks && n_warp + 4 * lane < n_cols) b4 = *reinterpret_cast<const float4*>(p.bias + n_warp + 4 * lane);
        if (4 * lane < 32 * own_chunks) st_shared16(bias_row + 16 * lane, __float_as_uint(b4.x), __float_as_uint(b4.y), __float_as_uint(b4.z), __float_as_uint(b4.w));
        __syncwarp();
      }
      if (is_dx(EPI) && n_warp < n_cols) {
        if (p.relubits_prev != nullptr) {
          const uint32_t* words = p.relubits_prev + m * ((p.N + 31) / 32) + (n_warp >> 5);
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (row_ok && c < own_chunks && n_warp + 32 * c < n_cols) prev_bits[c] = words[c];
        }
        if (elect_one()) tma_store_wait_read<0>();      // the unit before has left the buffers
        __syncwarp();
        if (EPI == kDxGelu) {
          for (int c = 0; c < own_chunks; ++c) prefetch_z(p, m_warp, n_warp + 32 * c, lane, stage + c * kChunkBytes);
          asm volatile("cp.async.commit_group;" ::: "memory");
        }
      }
      if (is_dx(EPI) && p.db != nullptr) {
        for (uint32_t k = 0; k < quota && cs.group < sum_groups && ok; ++k) {
          column_sums_step(p, cs, shift, et);
          if (++cs.step < sum_steps) continue;
          // the group is through: two buffers, so that one meeting of the warps per group is enough
          float* red = reinterpret_cast<float*>(epi_smem + kRingBytes) + (cs.turn & 1) * kEpiWarps * 16;
          column_sums_warp(cs, shift, lane, red + (warp - 2) * 16);
          ok = warps_meet(smem_u32(&ctl->group[0]), cs.turn & 1, wc, lane);
          const int64_t col = ((int64_t)cs.group << shift) * 8 + et;
          if (ok && et < (8 << shift) && col < p.K) {
            float t = 0.0f;
#pragma unroll
            for (int i = 0; i < kEpiWarps; ++i) t += red[i * 16 + et];
            p.db[col] = t;
          }
          cs.group += gridDim.x;
          cs.step = 0;
          ++cs.turn;
        }
        if (!ok) break;
      }
      if (lane == 0) ok = mbar_wait2(smem_u32(&ctl->tmem_full[0]) + 8u * buf, (buf_phases >> buf) & 1u, wc, 64u);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      if (EPI == kDxGelu) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
      }
      tc_fence_after();
#pragma unroll 1
      for (int c0 = c_first; c0 < c_last; c0 += 32) {
        const int64_t n = w.n0 + c0;
        if (n >= n_cols || (EPI != kDwT && m_warp >= sched.M)) break;               // warp-uniform
        const int c = (c0 - c_first) >> 5;
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256 + c0);
        uint32_t r[32];
        if (!is_dx(EPI)) {
          tmem_ld32(taddr, r);
          tmem_ld_wait();
        }
        if (EPI == kDwT) {
          // a chunk may reach past the tile's width (bn is a multiple of 16) and past the last kept column
          epilogue_chunk_dwt(p, r, m, n, (int)min((int64_t)min(32, bn - c0), n_cols - n), row_ok, w.split);
        } else if (is_dx(EPI)) {
          const uint32_t bits = c == 0 ? prev_bits[0] : c == 1 ? prev_bits[1] : c == 2 ? prev_bits[2] : prev_bits[3];
          dx_chunk<EPI == kDxGelu>(&tmO, taddr, (int)m_warp, (int)n, lane, bits, stage + c * kChunkBytes);
        } else {
          uint32_t ab[16];
          const uint32_t bits = forward_chunk<EPI % 3, kSlots>(p, &tmO, &tmL, &tmZ, r, (int)m_warp, (int)n, lane, stage, bias_row + 128 * c, turn++, ab);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i == c) act_bits[i] = bits;
          if (EPI >= kFwdFill)                         // from the chunk's buffer of activations, as forward_chunk took it
            place_kept(p, ab, sr, (int)(n >> 5) & 3, fill, stage + chunk_slot<kSlots>(turn - 1, p.out_zlow != nullptr) * kChunkBytes, lane);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(empty_bar + 8u * buf);
      if (is_forward(EPI)) {
        if (EPI >= kFwdFill && sr.staged) {              // all warps of the tile or none
          ok = group_sync();
          if (!ok) break;
          copy_kept(p, sr, fill, group_thread, 32 * group);
          ok = group_sync();
          if (!ok) break;
        }
        if (p.relubits != nullptr && row_ok && n_warp < n_cols) {
          uint32_t* words = p.relubits + m * p.w32 + (n_warp >> 5);
          if (own_chunks == 4 && p.w32 % 4 == 0 && n_warp + 96 < n_cols && ((uintptr_t)words & 15) == 0) {
            *reinterpret_cast<uint4*>(words) = make_uint4(act_bits[0], act_bits[1], act_bits[2], act_bits[3]);
          } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (c < own_chunks && n_warp + 32 * c < n_cols) words[c] = act_bits[c];
          }
        }
      }
      buf_phases ^= 1u << buf;
      buf ^= 1;
    }
    if (EPI != kDwT) {
      // a unit that was given up may have left z on its way
      if (EPI == kDxGelu) asm volatile("cp.async.wait_all;" ::: "memory");
      if (elect_one()) tma_store_wait();               // the results are out, and the buffers no longer read
      __syncwarp();
    }
  }

  // ===== teardown: neither CTA leaves (or frees tensor memory) while the other may still use it =====
  tc_fence_before();
  cluster_barrier();
  if (tid == 0 && ctl->abort_flag != 0) raise_status(p.dev_status, RAD_DEV_ETIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
  if (EPI != kDwT && p.beside && tid == 0) wait_for_previous();      // the kernels behind wait for this one's end: not before its elder's
}

// ---- two-CTA engine, sparse A (different-sample dW) --------------------------------------------------
// The pair owns a 256 x 512 tile of dW (narrower tiles take the first of the two halves, or half of that).  Each CTA rebuilds 128 columns of A_hat (one store tile per
// K block) in shared memory and loads its half of the dZ tile (two blocks of 128 columns); per 16
// rows of K two MMAs (M256 N256), one per 256-column half of the tile; the two 128 x 256
// accumulators of a CTA fill its tensor memory.  A store tile is expanded once per 512 output
// columns: the wide tile halves the expansion work per flop against a 256-column tile and brings the
// shared-memory traffic per K block and CTA from about 1540 to about 1200 wavefronts.
// Roles per CTA: 0 dZ producer, 1 MMA issuer (even CTA) and tensor-memory owner, 2-5 epilogue,
// 6 producer of the compressed ring, 7-22 expanders (two groups on alternate K blocks).  full[s] lives in the even CTA: one arrival
// with the dZ bytes of both CTAs plus one per expander warp of either CTA.
constexpr int kSpBM = 256, kSpBN = 512;      // widest tile: see plan_dw
constexpr int kSpAStageBytes = 128 * BK * 2;           // 16 KB: this CTA's 128 columns of A_hat
constexpr int sparse_stage_bytes(int bn) { return kSpAStageBytes + bn / 2 * BK * 2; }    // and this CTA's bn / 2 columns of dZ
constexpr int kSpMaxStages = 6;
constexpr int kSpExpanderWarps = 8;                    // per K block: one thread per keep-bit word of the store tile
constexpr int kSpExpanderGroups = 2;                   // groups of eight warps take alternate K blocks
constexpr int kSpEpiShare = 1 + kSpExpanderWarps * kSpExpanderGroups / 4;   // warps of a lane quarter that share the epilogue
constexpr int kSpThreads = 32 * (kFirstExpanderWarp + kSpExpanderGroups * kSpExpanderWarps);

struct SmemCtlSp {
  uint64_t full[kSpMaxStages], empty[kSpMaxStages], comp_full[8], comp_empty[8], tmem_full, tmem_empty;
  uint32_t tmem_base;
  int abort_flag;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSpThreads, 1)
tc_sparse_pair_kernel(const TcParams p, const __grid_constant__ CUtensorMap tmB) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int stages = p.num_stages, bn = p.bn;       // tile of 512 columns (two MMAs per 16 rows of K), 256 or 128
  const int stage_bytes = kSpAStageBytes + bn / 2 * BK * 2;
  const int comp_slot = kIndexBytes + p.comp_cap;               // index data + values of this CTA's store tile of one K block
  uint8_t* comp_base = smem + (size_t)stages * stage_bytes;
  SmemCtlSp* ctl = reinterpret_cast<SmemCtlSp*>(comp_base + (size_t)p.comp_depth * comp_slot);
  volatile int* abort_flag = &ctl->abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const uint32_t peer_abort = map_to_cta(smem_u32(&ctl->abort_flag), rank ^ 1u);
  const PairWait wc = {abort_flag, peer_abort, p.wait_limit_ns};
  const Schedule sched(p.M, p.N, p.K, p.splits, kSpBM, bn);
  const uint32_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  if (tid == 0) {
    prefetch_map(&tmB);
    for (int s = 0; s < stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1 + 2 * kSpExpanderWarps);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int c = 0; c < p.comp_depth; ++c) {
      mbar_init(smem_u32(&ctl->comp_full[c]), 1);
      mbar_init(smem_u32(&ctl->comp_empty[c]), kSpExpanderWarps);
    }
    mbar_init(smem_u32(&ctl->tmem_full), 1);
    mbar_init(smem_u32(&ctl->tmem_empty), 2 * 4 * kSpEpiShare);      // epilogue and expander warps of both CTAs
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&ctl->tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_barrier();
  tc_fence_after();
  const uint32_t tmem_base = ctl->tmem_base;
  const uint32_t smem_base = smem_u32(smem);
  // so far nothing of another kernel was touched: the above runs under the tail of the kernel before
  wait_for_previous();
  // this CTA's store tile column (128 columns of the layer input) of a unit, and whether it exists
  auto tile_col_of = [&](const Unit& w) -> int64_t { return (w.m0 + 128 * (int64_t)rank) / kTileCols; };
  // A warp's part of a unit's epilogue: 32-column chunks `first`, first + kSpEpiShare, ... of its lane quarter's rows
  auto unit_epilogue = [&](const Unit& w, int first, uint32_t parity) -> bool {
    const int q = warp & 3;
    bool ready = true;
    if (lane == 0) ready = mbar_wait2(smem_u32(&ctl->tmem_full), parity, wc, 100u);
    ready = __shfl_sync(0xffffffffu, ready ? 1 : 0, 0) != 0;
    if (!ready) return false;
    tc_fence_after();
    const int64_t m0 = w.m0 + 128 * (int64_t)rank + q * 32;
#pragma unroll 1
    for (int c0 = first * 32; c0 < bn; c0 += kSpEpiShare * 32) {
      const int64_t n = w.n0 + c0;
      if (n >= p.N) break;                  // warp-uniform
      epilogue_dw(p, tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, m0, n, w.split, lane);
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_remote(map_to_cta(smem_u32(&ctl->tmem_empty), 0u));
    return true;
  };

  if (warp == 0) {
    // ===== dZ producer: this CTA's 128 columns of each 256-column half of the dZ tile =====
    if (elect_one()) {
      const uint32_t full0 = map_to_cta(smem_u32(&ctl->full[0]), 0u);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
        const Unit w = sched.unit(u);
        if (u + npairs >= sched.units) let_next_start();
        const int n_own = (int)w.n0 + min(bn, 256) / 2 * (int)rank;       // + 256 for the second half
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          ok = mbar_wait2(smem_u32(&ctl->empty[0]) + 8u * stage, phase ^ 1u, wc);
          if (!ok) break;
          const uint32_t sB = smem_base + stage * stage_bytes + kSpAStageBytes;
          if (rank == 0) mbar_arrive_expect_tx(smem_u32(&ctl->full[0]) + 8u * stage, (uint32_t)bn * BK * 2);   // both CTAs' bytes
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (c * 128 < bn) tma_load_2d_pair(sB + c * 8192, &tmB, n_own + (c >> 1) * 256 + (c & 1) * 64, kb * BK, full0 + 8u * stage);
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
      }
      // every commit aimed at this CTA's stage barriers has landed before the CTA may leave
      for (int i = 0; i < stages && ok; ++i) {
        ok = mbar_wait2(smem_u32(&ctl->empty[0]) + 8u * stage, phase ^ 1u, wc);
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ===== MMA issuer (even CTA) =====
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = make_idesc_pair(true, true, (uint32_t)min(bn, 256));
      const bool halves = bn > 256;
      const uint64_t adesc0 = make_desc(smem_base, 8192, 1024), bdesc0 = make_desc(smem_base + kSpAStageBytes, 8192, 1024);
      int stage = 0;
      uint32_t phase = 0, unit_phase = 0;
      bool ok = true;
      for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
        const Unit w = sched.unit(u);
        ok = mbar_wait2(smem_u32(&ctl->tmem_empty), unit_phase ^ 1u, wc);
        if (!ok) break;
        tc_fence_after();
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          ok = mbar_wait2(smem_u32(&ctl->full[0]) + 8u * stage, phase, wc);
          if (!ok) break;
          tc_fence_after();
          const uint64_t adesc = adesc0 + (uint32_t)(stage * (stage_bytes >> 4));
          const uint64_t bdesc = bdesc0 + (uint32_t)(stage * (stage_bytes >> 4));
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
#pragma unroll
            for (int j = 0; j < 2; ++j)
              if (j == 0 || halves)
                tc_mma_pair(tmem_base + j * 256, adesc + k * (2048 >> 4), bdesc + (j * 16384 + k * 2048) / 16, idesc,
                            (kb > w.kb0 || k > 0) ? 1u : 0u);
          tc_commit_pair(smem_u32(&ctl->empty[0]) + 8u * stage);
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
        if (ok) tc_commit_pair(smem_u32(&ctl->tmem_full));
        unit_phase ^= 1u;
      }
    }
    __syncwarp();
  } else if (warp < 6) {
    // ===== epilogue: a warp = 32 accumulator rows, every kSpEpiShare-th 32-column chunk (the expanders take the others) =====
    uint32_t unit_phase = 0;
    bool ok = true;
    for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
      ok = unit_epilogue(sched.unit(u), 0, unit_phase);
      unit_phase ^= 1u;
    }
  } else if (warp == 6) {
    // ===== producer of the compressed ring: keep bits + row offsets (1152 B) and packed values of
    // this CTA's store tile of each K block.  It runs ahead of the A/B ring: a slot is free as soon
    // as the expanders have read it, long before the MMAs of that K block retire. =====
    int slot = 0;
    uint32_t cphase = 0;
    bool ok = true;
    for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
      const Unit w = sched.unit(u);
      const int64_t tile_col = tile_col_of(w);
      const bool have = tile_col < p.ncb;
      uint32_t off_lo = 0, off_hi = 0;                // tile offsets of K block (base + lane)
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        if (((kb - w.kb0) & 31) == 0 && have) {
          const int kbl = kb + lane;
          if (kbl < w.kb1) {
            const int64_t t0 = (int64_t)kbl * p.ncb + tile_col;
            off_lo = p.offsets[t0];
            off_hi = p.offsets[t0 + 1];
          }
        }
        const int src = (kb - w.kb0) & 31;
        const uint32_t o0 = __shfl_sync(0xffffffffu, off_lo, src);
        const uint32_t o1 = __shfl_sync(0xffffffffu, off_hi, src);
        bool sent = true;
        if (elect_one()) {
          sent = mbar_wait2(smem_u32(&ctl->comp_empty[slot]), cphase ^ 1u, wc);
          if (sent) {
            const uint32_t cfull = smem_u32(&ctl->comp_full[slot]);
            const uint32_t sC = smem_u32(comp_base) + slot * comp_slot;
            uint32_t vb = 0;
            if (have) {
              if (!tile_in_order(o0, o1)) raise_status(p.dev_status, RAD_DEV_EINTERNAL);          // no store's offsets
              else if (!tile_fits(o0, o1, p.values_capacity, (uint32_t)p.comp_cap)) raise_status(p.dev_status, RAD_DEV_ECAPACITY);
              else vb = (o1 - o0) * 2u;
            }
            mbar_arrive_expect_tx(cfull, (have ? (uint32_t)kIndexBytes : 0u) + vb);
            if (have) {
              bulk_load(sC, p.keepbits + ((int64_t)kb * p.ncb + tile_col) * kTileWords, kIndexBytes, cfull);
              if (vb != 0) bulk_load(sC + kIndexBytes, p.values + o0, vb, cfull);
            }
          }
        }
        ok = __all_sync(0xffffffffu, sent);
        if (!ok) break;
        if (++slot == p.comp_depth) { slot = 0; cphase ^= 1u; }
      }
    }
  } else {
    // ===== expanders: rebuild this CTA's A_hat tile (64 K rows x 128 columns, M-major, swizzled) =====
    // One thread per keep-bit word: row r of the slab, columns 32*wq..32*wq+31 of the store tile.
    // The row's first value is given by the stored row offset; the words before this one in the row
    // are counted with popc.  Eight consecutive lanes take eight consecutive rows of the same word
    // column: with the 128-byte swizzle their 16-byte zero stores then fall on eight different bank
    // groups.
    // Two groups of eight warps take alternate K blocks, so the waits, loads and fence of one K
    // block overlap the stores of the next.
    const int et = tid - 32 * kFirstExpanderWarp;            // 0..511
    const uint32_t group = (uint32_t)(et >> 8);
    const int wi = et & 255;
    const int r = (wi & 7) + ((wi >> 5) << 3), wq = (wi >> 3) & 3;
    int stage = 0, slot = 0;
    uint32_t phase = 0, cphase = 0, turn = 0, unit_phase = 0;
    bool ok = true;
    for (uint32_t u = pair; u < sched.units && ok; u += npairs) {
      const Unit w = sched.unit(u);
      const bool have = tile_col_of(w) < p.ncb;
      for (int kb = w.kb0; kb < w.kb1; ++kb, turn ^= 1u) {
        if (turn == group) {
          ok = mbar_wait2(smem_u32(&ctl->comp_full[slot]), cphase, wc) &&
               mbar_wait2(smem_u32(&ctl->empty[stage]), phase ^ 1u, wc);     // A tile of this stage is free
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          // columns past the layer's width keep whatever the buffer held: their accumulator rows are never written
          if (have) {
            uint8_t* sA = smem + (size_t)stage * stage_bytes;
            const uint8_t* sC = comp_base + (size_t)slot * comp_slot;
            expand_word(sA, sC, 0, r, wq, (uint32_t)p.comp_cap >> 1);
            fence_proxy_async();
          }
          __syncwarp();
          if (lane == 0) {
            mbar_arrive_remote(map_to_cta(smem_u32(&ctl->full[stage]), 0u));
            mbar_arrive(smem_u32(&ctl->comp_empty[slot]));
          }
        }
        if (++stage == stages) { stage = 0; phase ^= 1u; }
        if (++slot == p.comp_depth) { slot = 0; cphase ^= 1u; }
      }
      // The next unit's MMAs wait for this unit's accumulators to be read.  Sharing that is worth more than rebuilding the
      // next unit's first tiles meanwhile: 1024 x 8192 x 8192 140 us against 147 with the expanders ahead instead (and
      // sharing the last unit only), 2048 x 4096 x 4096 67 against 68, 8192 x 4096 x 4096 209 against 210.
      if (ok) ok = unit_epilogue(w, 1 + (warp - kFirstExpanderWarp) / 4, unit_phase);
      unit_phase ^= 1u;
    }
  }

  // ===== teardown: neither CTA leaves (or frees tensor memory) while the other may still use it =====
  tc_fence_before();
  cluster_barrier();
  if (tid == 0 && ctl->abort_flag != 0) raise_status(p.dev_status, RAD_DEV_ETIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// The pair kernels' bounded wait on a barrier nobody arrives at, in a cluster of two CTAs that owns no tensor
// memory and has no loads in flight: both waits run out, both abort flags go up, the pair meets at the
// cluster barrier as the real kernels do on their way out, and the status word reports the timeout.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(64, 1) wait_probe_pair_kernel(uint64_t limit_ns, int32_t* dev_status) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  const uint32_t rank = cluster_ctarank();
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cluster_barrier();
  const PairWait wc = {&abort_flag, map_to_cta(smem_u32(&abort_flag), rank ^ 1u), limit_ns};
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait2(smem_u32(&bar), 0u, wc, 100u);
  cluster_barrier();
  if (threadIdx.x == 0 && (!ok || abort_flag != 0)) raise_status(dev_status, RAD_DEV_ETIMEOUT);
}

// Sum of the K-split partial tiles in split order; rows may be scattered (same-sample).
__global__ void __launch_bounds__(256) dw_reduce_kernel(const float* partial, int64_t partial_rows, int splits,
                                                        int64_t M, const int64_t* M_dev, int64_t N,
                                                        const uint32_t* row_idx, float* out, int64_t ldw) {
  begin_after_previous();
  if (M_dev != nullptr) M = min(M, *M_dev);
  const int64_t n4 = N / 4, total = M * n4;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = i / n4, c = i % n4;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < splits; ++s) {
      const float4 v = __ldcs(reinterpret_cast<const float4*>(partial + ((int64_t)s * partial_rows + m) * N) + c);
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    const int64_t row = row_idx != nullptr ? (int64_t)row_idx[m] : m;
    reinterpret_cast<float4*>(out + row * ldw)[c] = acc;
  }
}

// ---- host side -------------------------------------------------------------------------------------
}  // namespace

// cuTensorMapEncodeTiled through the runtime's driver entry point table (no link against libcuda).
void* tensor_map_encoder() {
  static void* fn = nullptr;
  if (fn == nullptr) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = sym;
  }
  return fn;
}

namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() { return reinterpret_cast<EncodeTiledFn>(tensor_map_encoder()); }

// bf16 matrix, `inner` contiguous elements per row, `outer` rows of `ld` elements; box = 64 x box_outer.
int make_map(CUtensorMap* map, const void* ptr, int64_t inner, int64_t outer, int64_t ld, int box_outer) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return RAD_ECUDA;
  const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)box_outer};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? RAD_OK : RAD_ECUDA;
}

// Output matrix of `cols` x `rows` elements (bf16 or float32), stored in chunks of 32 x 32.
int make_out_map(CUtensorMap* map, bool f32, void* ptr, int64_t cols, int64_t rows, int64_t ld) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return RAD_ECUDA;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * (f32 ? 4 : 2)};
  const cuuint32_t box[2] = {32, 32};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ptr, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, f32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                        CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? RAD_OK : RAD_ECUDA;
}

int num_sms() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
      n = kNumSMsDefault;
  }
  return n;
}

// K splits of a same-sample dW.  Cost model in units of one CTA working through one K block
// (about 1024 tensor-pipe clocks): waves x K blocks per unit, plus what writing and re-reading the
// float32 partial tiles costs at HBM speed.  Pure function of the shapes, so the workspace query
// and the launch agree.
int choose_splits(int64_t m_tiles, int64_t n_tiles, int64_t kblocks, int64_t bm = BM, int64_t sms = kNumSMsDefault,
                  int64_t bn = BN, double kblock_scale = 1.0) {
  const double kblock_us = 0.55 * kblock_scale;                             // 1024 clk at ~1.9 GHz for a 256-wide tile
  const double partial_us = (double)(m_tiles * bm) * (double)(n_tiles * bn) * 8.0 / 6.5e6;   // per split
  int best = 1;
  double best_cost = 1e300;
  for (int s = 1; s <= kMaxSplits && s <= kblocks; ++s) {
    const int64_t units = m_tiles * n_tiles * s;
    const double cost = (double)ceil_div(units, sms) * (double)ceil_div(kblocks, s) * kblock_us +
                        (s > 1 ? partial_us * s + 5.0 : 0.0);
    if (cost < best_cost - 1e-9) { best_cost = cost; best = s; }
  }
  return best;
}

// Tile width and K splits of a different-sample dW of D x H from B rows.  What bounds it: a K block costs its expansion, 0.58 us
// whatever the width (0.84 at half the entries), up to 512 columns, whose MMAs and loads take 0.6; the epilogue 1.2 us per 128
// columns (a SM stores 50 bytes per ns); a launch its start and end; partial tiles a second launch and their bytes.  So a
// wide tile where the units fill the chip, a narrow one where they do not (us, wide / chosen: 328 x 640 x 520 13.5 / 9.4,
// 1024 x 512 x 512 14.0 / 11.0, 1024 x 2048 x 2048 20.1 / 17.9, 2048 x 1024 x 4096 29.9 / 27.3; kept at 512: 4096 x 2048 x 2048
// 40.6 against 46.0 at 256).  A pure function of the shapes, so that the workspace query and the launch agree.
struct SparseTile { int bn, splits; };
SparseTile choose_sparse_tile(int64_t B, int64_t D, int64_t H, double keep, int64_t pairs) {
  const int64_t kblocks = ceil_div(B, BK), m_tiles = ceil_div(D, kSpBM);
  const double out_us = (double)(m_tiles * kSpBM) * (double)H * 4.0 / 7.5e6;
  SparseTile best = {kSpBN, 1};
  double best_cost = 1e300;
  for (int bn = kSpBN; bn >= 128; bn /= 2) {
    const double kblock_us = (bn == kSpBN ? 0.62 : 0.58) + 0.65 * std::max(0.0, keep - 0.1), epilogue_us = bn / 128 * 1.25;
    for (int s = 1; s <= kMaxSplits && s <= kblocks; ++s) {
      const double waves = (double)ceil_div(m_tiles * ceil_div(H, bn) * s, pairs);
      const double beyond_l2 = out_us * s > 14.0 ? 2.0 : 1.0;         // 100 MB: partial tiles go through memory
      const double cost = waves * ((double)ceil_div(kblocks, s) * kblock_us + epilogue_us) + (s > 1 ? 2.5 + out_us * (s + 1) * beyond_l2 : 0.0);
      if (cost < best_cost - 1e-9) { best_cost = cost; best = {bn, s}; }
    }
  }
  return best;
}

struct DwPlan { int bn; int splits; int64_t partial_rows; int64_t bytes; int comp_cap; int stages; int comp_depth; };

// Clusters of two CTAs of `kernel` that can be resident at once.
template <typename K>
int resident_pairs_of(K kernel, int threads, size_t smem) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (num_sms() / 2));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n <= 0) {
    (void)cudaGetLastError();
    n = num_sms() / 2;
  }
  return std::min(n, num_sms() / 2);
}

// SM pairs the K splits of a dW contraction are planned for: what the device can really keep resident (a part
// whose SM count per GPC is odd somewhere hosts fewer two-CTA clusters than half its SMs, and a plan for 74
// pairs on 72 runs an extra wave), or half the default SM count where there is no device to ask (size queries
// on a host without one).  Found once, so that workspace queries and launches agree.
int planning_pairs() {
  static int pairs = 0;
  if (pairs == 0) {
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) == cudaSuccess && major == 10 &&
        cudaFuncSetAttribute(tc_sparse_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess) {
      pairs = resident_pairs_of(tc_sparse_pair_kernel, kSpThreads, 227 * 1024);
    } else {
      (void)cudaGetLastError();
      pairs = kNumSMsDefault / 2;
    }
  }
  return pairs;
}

DwPlan plan_dw(const rad_store* st, int64_t H) {
  DwPlan d = {};
  const int64_t kblocks = ceil_div(st->B, BK);
  int64_t m_expect;
  if (st->variant == RAD_SAME_SAMPLE) {
    // transposed tile: M = H, N = kept columns in tiles of at most 256 (the kernel fits the width to the count)
    m_expect = std::max<int64_t>(1, (int64_t)std::llround((double)st->D * store_keep_fraction(st)));
    d.partial_rows = round_up(std::min(st->values_ld, round_up(st->D, 8)), 16);
    const int64_t n_tiles = ceil_div(m_expect, BN);
    const int64_t bn = round_up(ceil_div(m_expect, n_tiles), 16);
    d.splits = choose_splits(ceil_div(H, BM), n_tiles, kblocks, BM, planning_pairs(), bn, (double)bn / BN);
    d.bytes = d.splits > 1 ? (int64_t)d.splits * d.partial_rows * H * 4 : 0;
    return d;
  } else {
    m_expect = st->D;
    d.partial_rows = round_up(st->D, BM);
    // per-tile value staging: mean + 8 sigma of Binomial(8192, p_eff), padded, in bytes
    const double pe = store_keep_fraction(st), n = (double)kTileRows * kTileCols;
    int64_t cap = (int64_t)(n * pe + 8.0 * std::sqrt(n * pe * (1.0 - pe)) + 16.0);
    cap = std::min<int64_t>(round_up(cap, 8), (int64_t)n) * 2;
    d.comp_cap = (int)round_up(cap, 128);
    const SparseTile tile = choose_sparse_tile(st->B, st->D, H, pe, planning_pairs());
    d.bn = tile.bn;
    d.splits = tile.splits;
    // shared memory: the A/B stages (48 KB for a tile of 512 columns) plus a ring of compressed slots
    const int64_t budget = 227 * 1024 - 2048 - (int64_t)sizeof(SmemCtlSp);
    const int64_t slot = kIndexBytes + d.comp_cap, stage = sparse_stage_bytes(d.bn);
    d.stages = kSpMaxStages;
    while (d.stages > 2 && d.stages * stage + (d.stages > 3 ? 3 : 2) * slot > budget) --d.stages;
    d.comp_depth = (int)std::max<int64_t>(2, std::min<int64_t>(8, (budget - d.stages * stage) / slot));
    d.bytes = d.splits > 1 ? (int64_t)d.splits * d.partial_rows * H * 4 : 0;
    return d;
  }
}

struct OutMaps { CUtensorMap o, l, z; };      // see tc_gemm_pair_kernel; those of absent outputs are not written through

template <int AK, int BKIND, int EPI, int kEpiWarps = 8>
int launch_pair(const TcParams& params, const CUtensorMap& ta, const CUtensorMap& tb, const OutMaps& out, int64_t max_units, cudaStream_t s) {
  TcParams p = params;
  const int stage = stage2_bytes(BKIND, EPI == kDwT ? BN : p.bn), rest = epi_bytes(EPI) + (int)sizeof(SmemCtl2) + 1024;
  p.num_stages = std::min(kStages2, (227 * 1024 - rest) / stage);
  const size_t smem = (size_t)p.num_stages * stage + rest;
  auto kernel = tc_gemm_pair_kernel<AK, BKIND, EPI, kEpiWarps>;
  // The kernel is persistent: the grid must not exceed the clusters that can be resident at once
  // (SM pairs that can host a cluster; fewer than half the SM count on some parts).
  static int resident_pairs = 0;
  if (resident_pairs == 0) {
    RAD_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    resident_pairs = resident_pairs_of(kernel, threads2(kEpiWarps), 227 * 1024);
  }
  const int pairs = (int)std::max<int64_t>(1, std::min<int64_t>(max_units, resident_pairs));
  count_launch();
  RAD_TRY(launch_kernel(kernel, 2 * pairs, threads2(kEpiWarps), smem, s, p, ta, tb, out.o, out.l, out.z));
  return RAD_OK;
}

int launch_sparse_pair(const TcParams& p, const CUtensorMap& tb, int64_t max_units, cudaStream_t s) {
  const size_t smem = (size_t)p.num_stages * sparse_stage_bytes(p.bn) + (size_t)p.comp_depth * (kIndexBytes + p.comp_cap) +
                      sizeof(SmemCtlSp) + 1024;
  if (smem > 227 * 1024 || p.num_stages > kSpMaxStages || p.comp_depth > 8) return RAD_EUNSUPPORTED;
  static int resident_pairs = 0;
  if (resident_pairs == 0) {
    RAD_CUDA_TRY(cudaFuncSetAttribute(tc_sparse_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    resident_pairs = resident_pairs_of(tc_sparse_pair_kernel, kSpThreads, 227 * 1024);
  }
  const int pairs = (int)std::max<int64_t>(1, std::min<int64_t>(max_units, resident_pairs));
  count_launch();
  RAD_TRY(launch_kernel(tc_sparse_pair_kernel, 2 * pairs, kSpThreads, smem, s, p, tb));
  return RAD_OK;
}

// Columns of an output tile of the forward pass and the input gradient: the narrowest of 64, 128 and 256 with which
// the tiles are still one wave of SM pairs, else 256.  Per K block an MMA of 256 columns takes 0.27 us, one of 64 or 128 with
// its loads 0.17 to 0.2: within a wave a narrower tile is no slower there and spreads loads and epilogues over more SMs
// (2048 x 1024 x 1024 forward with store: 21.8 / 16.9 / 22.0 us at 256 / 128 / 64 columns, which are 32 / 64 / 128 tiles on
// 74 pairs), a second wave costs most of the contraction again (4096 x 1024 x 1024: 22.2 / 25.0 / 36.1; both before the
// single-thread roles were elected).  A tile is no wider than the matrix needs either, or its stages are few and half empty (forward
// of 32768 x 4096 to 64 columns: 64.5 us in tiles of 256 columns and four stages, 49.2 now), but at least 128 where a store is filled, whose
// entries are staged by tiles of that width.
int dense_tile_width(int64_t M, int64_t N, int least = 64) {
  for (int bn = 64; bn < BN; bn *= 2)
    if (ceil_div(M, BM) * ceil_div(N, bn) <= planning_pairs() || (N <= bn && bn >= least)) return bn;
  return BN;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

}  // namespace

int launch_wait_probe_pair(uint64_t limit_ns, int32_t* dev_status, cudaStream_t s) {
  count_launch();
  wait_probe_pair_kernel<<<2, 64, 0, s>>>(limit_ns, dev_status);
  return cudaGetLastError() == cudaSuccess ? RAD_OK : RAD_ECUDA;
}

bool tc_shape_ok(int64_t B, int64_t D, int64_t H, const void* p0, int64_t ld0, const void* p1, int64_t ld1) {
  if (B < 64 || D < 64 || H < 64) return false;                    // tiny layers stay on CUDA cores
  if (D % 8 != 0 || H % 8 != 0) return false;
  if (!aligned16(p0) || !aligned16(p1) || ld0 % 8 != 0 || ld1 % 8 != 0) return false;
  if (B >= (1ll << 31) || D >= (1ll << 31) || H >= (1ll << 31)) return false;
  return encode_fn() != nullptr;
}
// Is it worth running such a contraction beside the kernel ahead?  Where its tiles leave SMs free: bf16 net 640-520-392-200, 328 rows
// 82.6 -> 73.4 us, four layers of 1024 at 4096 rows (128 tiles on 74 pairs) 226.6 and 226.3, at 8192 columns it only mixes operand streams.
static bool room_beside(int64_t units) { return units <= planning_pairs(); }

int tc_forward(int act, int64_t B, int64_t D, int64_t H, const void* A, int64_t lda, const void* W, int64_t ldw,
               const float* bias, void* out_act, int64_t ld_act, float* out_z, int64_t ld_z, void* out_zlow,
               int64_t ld_zlow, uint32_t* relubits, int32_t* dev_status, cudaStream_t s, const rad_store* next, bool beside) {
  CUtensorMap ta, tb;
  int rc = make_map(&ta, A, D, B, lda, 128);          // K-major A: box 64 (K) x 128 rows (one CTA of the pair)
  if (rc != RAD_OK) return rc;
  rc = make_map(&tb, W, H, D, ldw, 64);               // MN-major B: box 64 (N) x 64 K rows
  if (rc != RAD_OK) return rc;
  TcParams p = {};
  p.M = B; p.N = H; p.K = D; p.splits = 1; p.bn = dense_tile_width(B, H, next != nullptr ? 128 : 64);
  p.bias = bias;
  p.out_act = static_cast<const bf16*>(out_act); p.out_z = out_z; p.out_zlow = static_cast<const bf16*>(out_zlow);
  p.relubits = relubits; p.w32 = ceil_div(H, 32);
  p.dev_status = dev_status;
  p.wait_limit_ns = wait_limit_ns();
  if (next != nullptr) {
    // the store of this layer's output (B x H) as the next layer's input; its index part is in place
    if (out_act == nullptr || next->B != B || next->D != H || next->dtype != RAD_BF16 || !aligned16(next->keepbits))
      return RAD_EINVAL;
    p.st_values = static_cast<bf16*>(next->values); p.st_keepbits = next->keepbits; p.st_offsets = next->offsets;
    p.st_capacity = next->values_capacity; p.st_ncb = (int32_t)ceil_div(H, kTileCols);
    p.st_scale = next->law == RAD_LAW_FIXED ? (float)H / (float)draws_per_row_host(next->p, H)
                                            : (float)kLaneRange / (float)keep_threshold_host(next->p);
  }
  const int64_t units = ceil_div(B, BM) * ceil_div(H, p.bn);
  p.beside = beside && room_beside(units);
  OutMaps out = {};
  if (out_act != nullptr) RAD_TRY(make_out_map(&out.o, false, out_act, H, B, ld_act));
  if (out_zlow != nullptr) RAD_TRY(make_out_map(&out.l, false, out_zlow, H, B, ld_zlow));
  if (out_z != nullptr) RAD_TRY(make_out_map(&out.z, true, out_z, H, B, ld_z));
  // the kernel fetches a map ahead of time: each is one that was encoded
  if (out_act == nullptr) out.o = out_zlow != nullptr ? out.l : out.z;
  if (out_zlow == nullptr) out.l = out.o;
  if (out_z == nullptr) out.z = out.o;
  const bool fill = p.st_values != nullptr;
  const bool wide = fill ? D <= kWideEpilogueK
                         : act == RAD_ACT_GELU && D <= kWideGeluK && (out_zlow == nullptr || units <= kWideGeluWaves * planning_pairs());
  const auto launch = [&](auto epi) {
    constexpr int E = decltype(epi)::value;
    // without a store only a GELU has a form with sixteen warps
    if constexpr (E >= kFwdFill || E == kFwd + RAD_ACT_GELU)
      if (wide) return launch_pair<kAK, kBMN, E, 16>(p, ta, tb, out, units, s);
    return launch_pair<kAK, kBMN, E>(p, ta, tb, out, units, s);
  };
  switch (act + (fill ? kFwdFill : kFwd)) {
    case kFwd + RAD_ACT_RELU: return launch(std::integral_constant<int, kFwd + RAD_ACT_RELU>());
    case kFwd + RAD_ACT_GELU: return launch(std::integral_constant<int, kFwd + RAD_ACT_GELU>());
    case kFwdFill + RAD_ACT_NONE: return launch(std::integral_constant<int, kFwdFill + RAD_ACT_NONE>());
    case kFwdFill + RAD_ACT_RELU: return launch(std::integral_constant<int, kFwdFill + RAD_ACT_RELU>());
    case kFwdFill + RAD_ACT_GELU: return launch(std::integral_constant<int, kFwdFill + RAD_ACT_GELU>());
    default: return launch(std::integral_constant<int, kFwd>());
  }
}

// Whether the bias gradient goes beside the input gradient or into a launch of its own.  Beside it costs the CTAs of the
// contraction, however few, about 1.1 us per group of columns and 1.7 us per further step down the rows, of which each K block of
// their tiles hides 0.15 us; the launch costs 2.5 us and its reading.  Us, beside / separate: 4096 rows, dZ 1024 wide and inputs
// 1024 wide 11.0 / 17.5, 1024 x 8192 to 1024 28.0 / 35.5, but 256 x 4096 to 64 148 / 16, 16384 x 4096 to 256 101 / 70.  Over
// 238 shapes (64 to 16384 rows, 64 to 8192 columns) the choice is the faster one, or within 3 % of it but for five where it is
// within 8 %.
bool tc_sums_beside(int64_t B, int64_t D, int64_t H) {
  const int64_t bn = dense_tile_width(B, D), units = ceil_div(B, BM) * ceil_div(D, bn);
  const int64_t pairs = std::min<int64_t>(units, planning_pairs());
  const int shift = sum_shift(H, 2 * pairs);
  const int64_t groups = ceil_div(ceil_div(H, 8ll << shift), 2 * pairs), steps = ceil_div(B, (int64_t)(kSumThreads >> shift) * kSumLoads);
  const double sums = (double)groups * (1.1 + 1.7 * (double)(steps - 1)), hidden = 0.15 * (double)(ceil_div(units, pairs) * ceil_div(H, BK));
  return sums <= hidden + 2.5 + (double)B * (double)H * 2.0 / 6e6;
}

int tc_input_grad(int64_t B, int64_t D, int64_t H, const void* dZ, int64_t ldz, const void* W, int64_t ldw,
                  const uint32_t* relubits_prev, const void* z_prev, int64_t ld_zprev, void* dZ_prev, int64_t ldp,
                  float* db, int32_t* dev_status, cudaStream_t s, bool beside) {
  CUtensorMap ta, tb;
  int rc = make_map(&ta, dZ, H, B, ldz, 128);         // K-major A (K = H)
  if (rc != RAD_OK) return rc;
  const int bn = dense_tile_width(B, D);
  rc = make_map(&tb, W, H, D, ldw, bn / 2);           // K-major B: rows d (N), K = H contiguous
  if (rc != RAD_OK) return rc;
  TcParams p = {};
  p.M = B; p.N = D; p.K = H; p.splits = 1; p.bn = bn;
  p.relubits_prev = relubits_prev; p.z_prev = static_cast<const bf16*>(z_prev); p.ld_zprev = ld_zprev;
  p.dz = static_cast<const bf16*>(dZ); p.ld_dz = ldz; p.db = db;
  p.dev_status = dev_status;
  p.wait_limit_ns = wait_limit_ns();
  OutMaps out = {};
  RAD_TRY(make_out_map(&out.o, false, dZ_prev, D, B, ldp));
  out.l = out.z = out.o;
  const int64_t units = ceil_div(B, BM) * ceil_div(D, bn);
  p.beside = beside && room_beside(units);
  return z_prev != nullptr ? launch_pair<kAK, kBK_, kDxGelu>(p, ta, tb, out, units, s)
                           : launch_pair<kAK, kBK_, kDx>(p, ta, tb, out, units, s);
}

int sm_pairs() { return planning_pairs(); }

int64_t tc_weight_grad_workspace(const rad_store* st, int64_t H) {
  if (st->dtype != RAD_BF16 || st->D % 8 != 0 || H % 8 != 0 || st->B < 64 || st->D < 64 || H < 64) return 0;
  return plan_dw(st, H).bytes;
}

int tc_weight_grad(const rad_store* st, const void* dZ, int64_t ldz, int64_t H, float* dW, int64_t ldw,
                   void* workspace, int64_t workspace_bytes, int32_t* dev_status, cudaStream_t s) {
  const DwPlan d = plan_dw(st, H);
  if (d.bytes > 0 && (workspace == nullptr || workspace_bytes < d.bytes || !aligned16(workspace))) return RAD_EWORKSPACE;
  if (!aligned16(st->keepbits) || !aligned16(st->values)) return RAD_EUNSUPPORTED;
  CUtensorMap ta, tb;
  int rc = make_map(&tb, dZ, H, st->B, ldz, 64);      // MN-major B: box 64 (N = h) x 64 K rows (b)
  if (rc != RAD_OK) return rc;
  TcParams p = {};
  p.N = H; p.K = st->B; p.splits = d.splits; p.bn = d.bn; p.num_stages = d.stages; p.comp_depth = d.comp_depth;
  p.out_dw = dW; p.ld_dw = ldw; p.dw_rows = st->D; p.partial = static_cast<float*>(workspace); p.partial_rows = d.partial_rows;
  p.dev_status = dev_status;
  p.wait_limit_ns = wait_limit_ns();
  if (st->variant == RAD_SAME_SAMPLE) {
    // dW[idx, :]^T = dZ^T A_c: A operand dZ (M = h, MN-major), B operand the gathered block A_c (N = kept
    // column, MN-major), K = minibatch rows; the tile lands transposed and is scattered by kept column
    const int64_t nmax = std::min(st->values_ld, round_up(st->D, 8));
    ta = tb;                                           // dZ: box 64 (h) x 64 K rows
    rc = make_map(&tb, st->values, st->values_ld, st->B, st->values_ld, 64);
    if (rc != RAD_OK) return rc;
    p.M = H; p.N = nmax; p.N_dev = st->nnz; p.row_idx = st->offsets; p.keep_cols = st->keepbits;
    const int64_t n_expect = std::max<int64_t>(1, (int64_t)std::llround((double)st->D * store_keep_fraction(st)));
    rc = launch_pair<kAMN, kBMN, kDwT>(p, ta, tb, OutMaps{tb, tb, tb}, ceil_div(H, BM) * ceil_div(std::min(n_expect, nmax), BN) * d.splits, s);
  } else {
    ta = tb;                                           // unused by the sparse-A kernel
    p.M = st->D;
    p.values = static_cast<const bf16*>(st->values); p.keepbits = st->keepbits; p.offsets = st->offsets;
    p.values_capacity = st->values_capacity; p.ncb = (int32_t)ceil_div(st->D, kTileCols); p.comp_cap = d.comp_cap;
    rc = launch_sparse_pair(p, tb, ceil_div(st->D, kSpBM) * ceil_div(H, d.bn) * d.splits, s);
  }
  if (rc != RAD_OK) return rc;
  if (d.splits > 1) {
    const int64_t rows = st->variant == RAD_SAME_SAMPLE ? p.N : p.M;       // rows of a partial block
    const int64_t work = rows * (H / 4);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(work, 256), 148 * 16));
    count_launch();
    RAD_TRY(launch_kernel(dw_reduce_kernel, grid, 256, 0, s, p.partial, d.partial_rows, d.splits, rows, p.N_dev, H, p.row_idx, dW, ldw));
  }
  return RAD_OK;
}

}  // namespace rad
