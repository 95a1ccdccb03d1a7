// CUDA-core (FFMA) kernels: small float32 contractions (larger ones go to gemm_tc.cu, three exact bf16 planes per operand) and
// bf16 problems whose shapes the TMA path cannot take.  These problems are latency-bound; the kernels favour exact float32
// accumulation in a fixed order over speed.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "gemm.cuh"

namespace rad {
namespace {

// Splitting a contraction over CTAs: the CTAs of a tile are neighbours in a cluster, each leaves its partial tile
// in its own shared memory, and each then finishes (adds in split order, applies the epilogue to, writes) an equal
// share of the tile's rows, reading the others' partial sums through distributed shared memory.
__device__ __forceinline__ void share_barrier() {
  if (cluster_nctas() > 1) cluster_barrier(); else __syncthreads();
}
__device__ __forceinline__ void copy_async16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy_async4(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}

constexpr int kGemmBK = 64;                          // k per block
constexpr int kGemmStages = 3;                       // float32: K blocks in flight or being multiplied
__host__ __device__ constexpr int gemm_operand_floats(int ts) { return ts * (kGemmBK + 4) > kGemmBK * (ts + 4) ? ts * (kGemmBK + 4) : kGemmBK * (ts + 4); }
__host__ __device__ constexpr int gemm_smem_bytes(int ts) { return kGemmStages * 2 * gemm_operand_floats(ts) * 4; }
constexpr int kGemmSmemBytes = gemm_smem_bytes(64);
static_assert(gemm_smem_bytes(32) >= 4 * 64 * (32 + 4) * 4, "the walking form fits the same buffer");
static_assert(gemm_smem_bytes(32) >= (4 * 32 * 32 + 32) * 4 && gemm_smem_bytes(64) >= (4 * 64 * 64 + 64) * 4,
              "the partial tiles and column sums reuse the ring");

// Asynchronous copies of one operand's K blocks into the ring, in the layout it has in memory: TS rows of BK
// contiguous k (kKM) or BK rows of TS contiguous columns, zeros outside the matrix and past the end of the split.
// A thread keeps one running pointer; everything that does not change from block to block is found once.
// kTurn: k is contiguous in memory, but the block lands as BK rows of TS columns (single elements).
template <bool kKM, bool kTurn, int TS, int BK>
struct BlockCopy {
  static constexpr int kInner = kKM ? BK : TS, kLds = kTurn ? TS + 4 : kInner + 4;
  static constexpr int kVec = TS * BK / 1024, kOne = TS * BK / 256;      // copies a thread makes per block
  const float* src; const float* safe;
  int64_t step, advance;
  int o, i, fixed; uint32_t ok;
  bool vec;
  __device__ __forceinline__ void init(const float* X, int64_t ld, int64_t r0, int64_t rows, int64_t k0, bool vec16) {
    vec = vec16 && !kTurn;
    const int per_row = vec ? kInner / 4 : kInner, w = vec ? 4 : 1, ostep = 256 / per_row;
    o = (int)threadIdx.x / per_row;
    i = ((int)threadIdx.x % per_row) * w;
    step = (int64_t)ostep * ld;
    safe = X;
    ok = 0;
    if (kKM) {
      for (int j = 0; j < kOne; ++j) ok |= (r0 + o + j * ostep < rows ? 1u : 0u) << j;
      fixed = w * 4;
      src = X + (r0 + o) * ld + k0 + i;
      advance = BK;
    } else {
      const int64_t left = rows - (r0 + i);
      fixed = left >= w ? w * 4 : left > 0 ? (int)left * 4 : 0;
      src = X + (k0 + o) * ld + r0 + i;
      advance = (int64_t)BK * ld;
    }
  }
  template <bool kV>
  __device__ __forceinline__ void copies(float* dst, int kleft) {
    constexpr int per_row = kV ? kInner / 4 : kInner, ostep = 256 / per_row, w = kV ? 4 : 1;
    float* d = kTurn ? dst + i * kLds + o : dst + o * kLds + i;
#pragma unroll
    for (int j = 0; j < (kV ? kVec : kOne); ++j) {
      int bytes;
      if (kKM) bytes = ((ok >> j) & 1u) != 0 ? min(max(kleft - i, 0), w) * 4 : 0;
      else bytes = o + j * ostep < kleft ? fixed : 0;
      const float* from = bytes != 0 ? src + j * step : safe;
      if (kV) copy_async16(d + j * ostep * kLds, from, bytes); else copy_async4(d + j * ostep * (kTurn ? 1 : kLds), from, bytes);
    }
  }
  __device__ __forceinline__ void issue(float* dst, int kleft) {         // kleft: k of the block inside the split, or more
    if (!kTurn && vec) copies<true>(dst, kleft); else copies<false>(dst, kleft);
    src += advance;
  }
};

// The A operand of a different-sample dW: K block = one slab of 64 rows of the store, TS of a store tile's 128 columns,
// expanded on the way into the ring (every entry is a four-byte copy, of nothing where it was not kept).  A thread
// takes every fourth column of one row, so that a warp's copies fall on all banks; a value's place is the row's
// offset plus the kept entries before it.  The index words of the next slab are in registers before they are needed.
// 1500 x 1001 x 777: 89 us at any keep probability, 172 (p = 0.1) to 385 us (p = 1) with a tile rebuilt by popcounts
// between two barriers and four scalar shared-memory reads per operand; 4096 x 128 x 10 bf16: 356 -> 19 us (its 64 slabs
// were one CTA's walk).  A walk over per-column lists of kept rows (no zeros multiplied) was slower from p = 0.1 up:
// 95 / 274 / 554 us at p = 0.1 / 0.5 / 1 on the first shape.
template <typename T, int TS>
struct SparseCopy {
  static constexpr int kWords = TS / 32;
  const uint32_t* tile; const uint32_t* offset; const T* values;
  int64_t capacity, tile_step; int ncb, w0, r, q;
  uint32_t word[kWords]; int64_t at[kWords];
  __device__ __forceinline__ void init(const GemmParams& p, int64_t m0, int64_t k0) {
    const int64_t t = k0 / kTileRows * p.ncb + m0 / kTileCols;
    r = (int)threadIdx.x >> 2; q = (int)threadIdx.x & 3;
    w0 = (int)(m0 % kTileCols) / 32;
    tile = p.keepbits + t * kTileWords; offset = p.offsets + t;
    ncb = p.ncb; tile_step = (int64_t)p.ncb * kTileWords;
    values = static_cast<const T*>(p.A); capacity = p.capacity;
  }
  __device__ __forceinline__ void load_index() {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = tile[4 * r + i];
    int64_t pos = (int64_t)*offset + ((tile[kBitWords + (r >> 1)] >> (16 * (r & 1))) & 0xffffu);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int j = 0; j < kWords; ++j)
        if (i == w0 + j) { word[j] = w[i]; at[j] = pos; }
      pos += __popc(w[i]);
    }
    tile += tile_step; offset += ncb;
  }
  // place of element j (column q + 4 j of the TS), or -1 where it was not kept or lies past the store's capacity
  __device__ __forceinline__ int64_t place(int j) const {
    const uint32_t bit = 1u << (q + 4 * (j & 7));
    const int64_t pos = at[j >> 3] + __popc(word[j >> 3] & (bit - 1));
    return (word[j >> 3] & bit) != 0 && pos < capacity ? pos : -1;
  }
};

// One CTA's share of a TS x TS tile of C (256 threads).  Four groups of 64 threads take every fourth quartet of k of
// a 64-deep K block; a thread of a group owns TS/8 x TS/8 outputs; the groups' tiles are added at the end.  float32
// operands arrive through a three-deep ring of asynchronous copies (zero-filled outside the matrix), bf16 ones are
// widened on the way through registers one block ahead.  B lies k-major in shared memory whichever way round it
// is in memory: pairs of columns feed the paired multiply-adds without being assembled (the input gradient of
// 4096 x 2048 x 2048: 1438 us with pairs assembled from rows, 865 with single-element copies that turn the block).
// What bounds it: the FMA pipes and register file for layers that fill the chip (that input gradient: 1221 us
// before; the forward pass 1175 -> 806 us, 43 TFLOP/s), else the latency of the chain load -> multiply -> add, so k
// is split over the groups and up to eight CTAs (150 x 300 outputs, k = 784: 23.2 -> 9.3 us).  Sums over the groups and
// splits are also several times shorter chains of roundings than one thread's walk along k.
template <typename T, int EPI, int TS>
__device__ __forceinline__ void gemm_partial(const GemmParams& p, int tile, int split, float* smem) {
  constexpr bool kSparse = EPI == kEpiSparse;
  constexpr bool kAK = EPI == kEpiForward || EPI == kEpiInputGrad, kBK = EPI == kEpiInputGrad;      // k contiguous in memory?
  constexpr int BK = kGemmBK, TM = TS / 8;
  constexpr int kLdA = kAK ? BK + 4 : TS + 4, kLdB = TS + 4;                    // 16-byte multiples, conflict-free
  constexpr int kGemmStageFloats = 2 * gemm_operand_floats(TS);
  // what only needs the parameters is done before the kernel ahead has ended (MNIST-shaped step of ten launches 70.2 -> 66 us)
  int64_t M = p.M;
  if (EPI == kEpiScatterRows) {
    begin_after_previous();
    if (p.M_dev != nullptr) M = min(M, *p.M_dev);
  }
  const int gx = (int)p.gx;
  const int64_t m0 = (int64_t)(tile / gx) * TS, n0 = (int64_t)(tile % gx) * TS;
  const bool sums = (EPI == kEpiScatterRows || EPI == kEpiSparse) && p.db != nullptr && m0 == 0;
  if (m0 >= M && !sums) return;
  const int tid = threadIdx.x, group = tid >> 6, t = tid & 63, ty = t >> 3, tx = t & 7;
  const T* A = static_cast<const T*>(p.A);
  const T* Bm = static_cast<const T*>(p.Bm);
  const int64_t k0 = (int64_t)split * p.k_per, k1 = min(p.K, k0 + p.k_per);
  const int nblk = k1 > k0 ? (int)((k1 - k0 + BK - 1) / BK) : 0;
  f32x2 acc[TM][TM / 2] = {};                        // outputs in pairs of neighbouring columns j
  float colsum = 0.0f;
  BlockCopy<kAK, false, TS, BK> ca;
  BlockCopy<kBK, kBK, TS, BK> cb;
  SparseCopy<T, TS> cs;
  static_assert(!kSparse || BK == kTileRows, "a K block of a different-sample dW is a slab of the store");
  if constexpr (kSparse) cs.init(p, m0, k0);
  if constexpr (sizeof(T) == 4) {
    if (!kSparse) ca.init(reinterpret_cast<const float*>(A), kAK ? p.sam : p.sak, m0, M, k0, p.vec_a != 0);
    cb.init(reinterpret_cast<const float*>(Bm), kBK ? p.sbn : p.sbk, n0, p.N, k0, p.vec_b != 0);
  }
  if (EPI != kEpiScatterRows) begin_after_previous();
  if constexpr (kSparse) {
    if (nblk > 0) cs.load_index();
  }
  auto issue = [&](int kb) {
    if constexpr (sizeof(T) == 4) {
      if (kb < nblk) {
        float* sA = smem + (kb % kGemmStages) * kGemmStageFloats;
        const int kleft = (int)min((int64_t)BK, k1 - k0 - (int64_t)kb * BK);
        if constexpr (kSparse) {
#pragma unroll
          for (int j = 0; j < TS / 4; ++j) {
            const int64_t at = cs.place(j);
            copy_async4(sA + cs.r * kLdA + cs.q + 4 * j, reinterpret_cast<const float*>(cs.values) + (at >= 0 ? at : 0), at >= 0 ? 4 : 0);
          }
          if (kb + 1 < nblk) cs.load_index();
        } else {
          ca.issue(sA, kleft);
        }
        cb.issue(sA + kGemmStageFloats / 2, kleft);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  };
  constexpr int NF = TS * BK / 256;
  float ra[sizeof(T) == 2 ? NF : 1], rb[sizeof(T) == 2 ? NF : 1];
  auto fetch = [&](int kb) {
    if constexpr (sizeof(T) == 2) {
#pragma unroll
      for (int j = 0; j < NF; ++j) {
        const int c = tid + j * 256;
        if constexpr (kSparse) {
          const int64_t at = cs.place(j);
          ra[j] = at >= 0 ? to_float(cs.values[at]) : 0.0f;
        } else {
          const int64_t ma = m0 + (kAK ? c / BK : c % TS), ka = k0 + (int64_t)kb * BK + (kAK ? c % BK : c / TS);
          ra[j] = ma < M && ka < k1 ? to_float(A[ma * p.sam + ka * p.sak]) : 0.0f;
        }
        const int64_t nb = n0 + (kBK ? c / BK : c % TS), kk = k0 + (int64_t)kb * BK + (kBK ? c % BK : c / TS);
        rb[j] = nb < p.N && kk < k1 ? to_float(Bm[kk * p.sbk + nb * p.sbn]) : 0.0f;
      }
      if constexpr (kSparse) {
        if (kb + 1 < nblk) cs.load_index();
      }
    }
  };
  auto stash = [&](int kb) {
    if constexpr (sizeof(T) == 2) {
      float* sA = smem + (kb % kGemmStages) * kGemmStageFloats;
      float* sB = sA + kGemmStageFloats / 2;
#pragma unroll
      for (int j = 0; j < NF; ++j) {
        const int c = tid + j * 256;
        if (kSparse) sA[cs.r * kLdA + cs.q + 4 * j] = ra[j];
        else sA[(kAK ? c / BK : c / TS) * kLdA + (kAK ? c % BK : c % TS)] = ra[j];
        sB[(kBK ? c % BK : c / TS) * kLdB + (kBK ? c / BK : c % TS)] = rb[j];
      }
    }
  };
  if constexpr (sizeof(T) == 4) {
    for (int i = 0; i < kGemmStages - 1; ++i) issue(i);
  } else if (nblk > 0) {
    fetch(0);
    stash(0);
  }
  for (int kb = 0; kb < nblk; ++kb) {
    if constexpr (sizeof(T) == 4) asm volatile("cp.async.wait_group %0;" ::"n"(kGemmStages - 2) : "memory");
    __syncthreads();                                 // block kb is in place, and everyone is done with block kb - 1
    if constexpr (sizeof(T) == 4) issue(kb + kGemmStages - 1);
    else if (kb + 1 < nblk) fetch(kb + 1);
    const float* sA = smem + (kb % kGemmStages) * kGemmStageFloats;
    const float* sB = sA + kGemmStageFloats / 2;
    if (sums && tid < TS) {
      // the block of Bm is in shared memory anyway: its column sums, row after row (rows past k1 hold zeros)
#pragma unroll 8
      for (int kk = 0; kk < BK; ++kk) colsum += sB[kk * kLdB + tid];
    }
    auto quartet = [&](int kc) {
#pragma unroll
      for (int h = 0; h < 4; h += 2) {               // two k at a time
        float a[TM][2];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          if (kAK) {
            const float2 v = *reinterpret_cast<const float2*>(sA + (ty + 8 * i) * kLdA + kc + h);
            a[i][0] = v.x; a[i][1] = v.y;
          } else if (i % 4 == 0) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const float4 v = *reinterpret_cast<const float4*>(sA + (kc + h + k) * kLdA + ty * 4 + 8 * i);
              a[i][k] = v.x; a[i + 1][k] = v.y; a[i + 2][k] = v.z; a[i + 3][k] = v.w;
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          f32x2 bb[TM / 2];
#pragma unroll
          for (int j = 0; j < TM / 2; j += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(sB + (kc + h + k) * kLdB + tx * 4 + 16 * j);
            bb[j] = v.x; bb[j + 1] = v.y;
          }
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const f32x2 aa = pack2(a[i][k], a[i][k]);
#pragma unroll
            for (int j = 0; j < TM / 2; ++j) fma2(acc[i][j], aa, bb[j]);
          }
        }
      }
    };
    const int kvalid = (int)min((int64_t)BK, k1 - k0 - (int64_t)kb * BK);
    if (kvalid == BK) {
#pragma unroll
      for (int kc = 0; kc < BK; kc += 16) quartet(kc + group * 4);
    } else {
#pragma unroll 1
      for (int kc = group * 4; kc < kvalid; kc += 16) quartet(kc);
    }
    if constexpr (sizeof(T) == 2) {
      if (kb + 1 < nblk) stash(kb + 1);
    }
  }
  if constexpr (sizeof(T) == 4) asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  float* plane = smem + group * TS * TS;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; j += 2) {
      const int m = kAK ? ty + 8 * i : ty * 4 + (i & 3) + 32 * (i >> 2);
      const int n = tx * 4 + (j & 3) + 32 * (j >> 2);
      unpack2(acc[i][j / 2], plane[m * TS + n], plane[m * TS + n + 1]);
    }
  if (sums && tid < TS) smem[4 * TS * TS + tid] = colsum;
  __syncthreads();
#pragma unroll 4
  for (int e = tid; e < TS * TS; e += 256)
    smem[e] = (smem[e] + smem[TS * TS + e]) + (smem[2 * TS * TS + e] + smem[3 * TS * TS + e]);
}

// The CTA's share of the tile's rows, from the partial tiles of all its splits: a thread has one column and every 256 / TS-th row.
// What an output needs besides its sums is under way for four rows before the first is written.
template <typename T, int EPI, int TS>
__device__ __forceinline__ void gemm_finish(const GemmParams& p, int tile, int split, const float* smem) {
  int64_t M = p.M;
  if (p.M_dev != nullptr) M = min(M, *p.M_dev);
  const int gx = (int)p.gx;
  const int64_t m0 = (int64_t)(tile / gx) * TS, n0 = (int64_t)(tile % gx) * TS;
  const bool sums = (EPI == kEpiScatterRows || EPI == kEpiSparse) && p.db != nullptr && m0 == 0;
  const int S = p.splits, rows = TS / S, tid = threadIdx.x;
  const uint32_t rank0 = cluster_ctarank() - (uint32_t)split;
  if (sums && split == 0 && tid < TS && n0 + tid < p.N) {
    float s = 0.0f;
    for (int q = 0; q < S; ++q) s += S > 1 ? ld_cluster_f32(smem + 4 * TS * TS + tid, rank0 + q) : smem[4 * TS * TS + tid];
    p.db[n0 + tid] = s;
  }
  if (m0 >= M) return;
  constexpr int kStep = 256 / TS, kAhead = 4;
  const int c = tid % TS, end = (int)min((int64_t)(split + 1) * rows, M - m0);
  const int64_t n = n0 + c;
  if (n >= p.N) return;
  GemmSide side;
  side.bias = EPI == kEpiForward && p.bias != nullptr ? p.bias[n] : 0.0f;
#pragma unroll 1
  for (int r0 = split * rows + tid / TS; r0 < end; r0 += kAhead * kStep) {
    float v[kAhead], z[kAhead];
    uint32_t word[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int r = min(r0 + i * kStep, end - 1);
      gemm_prefetch<T, EPI>(p, m0 + r, n, word[i], z[i]);
      v[i] = S == 1 ? smem[r * TS + c] : 0.0f;
    }
#pragma unroll 8
    for (int q = 0; S > 1 && q < S; ++q) {
#pragma unroll
      for (int i = 0; i < kAhead; ++i) v[i] += ld_cluster_f32(smem + min(r0 + i * kStep, end - 1) * TS + c, rank0 + q);
    }
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      if (r0 + i * kStep >= end) break;
      side.word = word[i];
      side.z = z[i];
      gemm_store<T, EPI>(p, m0 + r0 + i * kStep, n, v[i], side);
    }
  }
}

// The other form, for short contractions and most bf16 shapes (see plan_gemm): one TS x TS tile of C by one CTA of 256
// threads that walks all of k, TS/16 x TS/16 outputs per thread, the next step's rows of K in registers while the
// current ones are multiplied out of shared memory; nothing to add at the end.  Every output is one chain of fused
// multiply-adds over k in ascending order.  K rows per step: the small tile takes four times as many, so that its
// steps, which are bound by the latency of their loads, are a quarter as many.
constexpr int walk_bk(int ts) { return ts == 32 ? 64 : 16; }
constexpr int walk_smem_bytes(int ts) { return 4 * walk_bk(ts) * (ts + 4) * 4; }
template <typename T, int EPI, int TS>
__device__ __forceinline__ void gemm_walk(const GemmParams& p, int64_t tile, float* smem) {
  constexpr int kBM = TS, kBN = TS, TM = TS / 16, kBK = walk_bk(TS), NF = TS * kBK / 256;
  constexpr int kLdS = TS + 4;                       // floats per k row of a staged operand (16-byte multiples)
  static_assert((kLdS * 4) % 16 == 0 && (TM == 4 || TM == 2), "vector reads of the staged operands");
  int64_t M = p.M;
  if (p.M_dev != nullptr) M = min(M, *p.M_dev);
  const int64_t m0 = tile / p.gx * kBM, n0 = tile % p.gx * kBN;
  const bool sums = EPI == kEpiScatterRows && p.db != nullptr && m0 == 0;
  if (m0 >= M && !sums) return;
  const int tid = threadIdx.x;
  float colsum = 0.0f;
  const int tm = (tid >> 4) * TM, tn = (tid & 15) * TM;
  const T* A = static_cast<const T*>(p.A);
  const T* Bm = static_cast<const T*>(p.Bm);
  float acc[TM][TM] = {};
  // TS x kBK elements of each operand per step; whichever index is contiguous in memory is made
  // the fast thread index
  float ra[NF], rb[NF];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int j = 0; j < NF; ++j) {
      const int i = tid + j * 256;
      int mm, kk;
      if (p.sak == 1) { kk = i % kBK; mm = i / kBK; } else { mm = i % kBM; kk = i / kBM; }
      const int64_t m = m0 + mm, k = k0 + kk;
      ra[j] = (m < M && k < p.K) ? to_float(A[m * p.sam + k * p.sak]) : 0.0f;
      int nn;
      if (p.sbk == 1) { kk = i % kBK; nn = i / kBK; } else { nn = i % kBN; kk = i / kBN; }
      const int64_t n = n0 + nn, kb = k0 + kk;
      rb[j] = (n < p.N && kb < p.K) ? to_float(Bm[kb * p.sbk + n * p.sbn]) : 0.0f;
    }
  };
  auto stash = [&](int buf) {
    float* sA = smem + buf * 2 * kBK * kLdS;
    float* sB = sA + kBK * kLdS;
#pragma unroll
    for (int j = 0; j < NF; ++j) {
      const int i = tid + j * 256;
      if (p.sak == 1) sA[(i % kBK) * kLdS + i / kBK] = ra[j]; else sA[(i / kBM) * kLdS + i % kBM] = ra[j];
      if (p.sbk == 1) sB[(i % kBK) * kLdS + i / kBK] = rb[j]; else sB[(i / kBN) * kLdS + i % kBN] = rb[j];
    }
  };
  fetch(0);
  stash(0);
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = 0; k0 < p.K; k0 += kBK) {
    const bool more = k0 + kBK < p.K;
    if (more) fetch(k0 + kBK);
    const float* sA = smem + buf * 2 * kBK * kLdS;
    const float* sB = sA + kBK * kLdS;
    if (sums && tid < kBN) {
      // the block of Bm is in shared memory anyway: its column sums, row after row (rows past K hold zeros)
#pragma unroll
      for (int kk = 0; kk < kBK; ++kk) colsum += sB[kk * kLdS + tid];
    }
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
      float a[TM], b[TM];
      if (TM == 4) {
        const float4 a4 = *reinterpret_cast<const float4*>(sA + kk * kLdS + tm);
        const float4 b4 = *reinterpret_cast<const float4*>(sB + kk * kLdS + tn);
        a[0] = a4.x; a[1] = a4.y; a[TM - 2] = a4.z; a[TM - 1] = a4.w;
        b[0] = b4.x; b[1] = b4.y; b[TM - 2] = b4.z; b[TM - 1] = b4.w;
      } else {
        const float2 a2 = *reinterpret_cast<const float2*>(sA + kk * kLdS + tm);
        const float2 b2 = *reinterpret_cast<const float2*>(sB + kk * kLdS + tn);
        a[0] = a2.x; a[1] = a2.y;
        b[0] = b2.x; b[1] = b2.y;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  if (sums && tid < kBN && n0 + tid < p.N) p.db[n0 + tid] = colsum;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t m = m0 + tm + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      const int64_t n = n0 + tn + j;
      if (n >= p.N) continue;
      gemm_store<T, EPI>(p, m, n, acc[i][j], gemm_side<T, EPI>(p, m, n));
    }
  }
}

// Tile and split of a contraction: the pair with the least estimated time, in clocks of the SM that gets the most
// CTAs.  Two CTAs share an SM; per k of its share a pair takes 106 clocks with 64 x 64 tiles and 35 with 32 x 32
// (0.60 and 0.46 of the FMA rate), a CTA alone 73 and 26; beginning and end of a CTA (first loads, the groups'
// sums, epilogue) take 7500 and 3850, the launch 4000, the exchange inside a cluster 800.  Fitted to 32 timings
// (both tiles, 1 to 8 splits); for 150 x 300 outputs it says 28 / 19 / 19 / 22 thousand clocks for 1 / 2 / 4 / 8 CTAs
// per 32 x 32 tile at k = 784, measured 26 / 19 / 18 / 23; for 1500 x 777, k = 1001, 105 / 95 / 101 us for 1 / 2 / 4 CTAs
// per 64 x 64 tile, measured 112 / 101 / 102.
// The walking form (no split, no sums at the end) is weighed with figures of its own, and bf16 operands, which both forms
// widen on the way through registers, with others again (the split form's depend on whether k is contiguous: more
// address arithmetic and spilled registers then).  So the walking form takes short contractions (4096 x 1001 f32, k =
// 10: 17 us against 34; the lines cross near k = 160 where the chip is full and near k = 80 where it is not) and bf16
// shapes that fill the chip (1024 x 1023 x 1021 forward: 95 against 137 us).  Checked with either form forced: of 120
// forwards, input gradients and same-sample dW of both types, 16 to 4096 rows, the choice is within 6 % of the better form in
// 118; the others are bf16 300 x 100 x 700 (forward 10.2 against 9.2 us, dW 16.9 against 13.9).
struct GemmCost { double pair, alone, ends; };
inline double plan_gemm(GemmParams& p, int64_t Mgrid, int es, int64_t k_step = 4, bool may_walk = true) {   // splits begin at multiples of k_step
  static const GemmCost split_cost[3][2] = {{{35, 26, 3850}, {106, 73, 7500}},      // f32, at 32 x 32 and 64 x 64
                                            {{72, 45, 4500}, {258, 150, 11000}},    // bf16, k contiguous
                                            {{72, 45, 4500}, {150, 90, 7500}}};     // bf16, dW
  static const GemmCost walk_cost[2][2] = {{{80, 46, 2000}, {158, 100, 3500}}, {{110, 72, 2000}, {168, 110, 3800}}};
  const int kind = es == 4 ? 0 : p.sak == 1 ? 1 : 2;
  double best = 1e300;
  for (int ts = 32; ts <= 64; ts *= 2) {
    const int64_t tiles = std::max<int64_t>(1, ceil_div(Mgrid, ts)) * ceil_div(p.N, ts);
    for (int s = may_walk ? 0 : 1; s <= 8; s = s == 0 ? 1 : 2 * s) {               // 0: the walking form
      if (s > 1 && (p.K < 16 * s || p.K <= s / 2 * k_step)) break;
      const int n = std::max(s, 1);
      const GemmCost& c = (s == 0 ? walk_cost[es == 2] : split_cost[kind])[ts == 64];
      const int64_t per_sm = ceil_div(tiles * n, 148), k_per = round_up(ceil_div(p.K, n), k_step);
      const double clk = (double)k_per * ((double)(per_sm / 2) * c.pair + (double)(per_sm % 2) * c.alone) + (double)per_sm * c.ends + 4000.0 +
                         (n > 1 ? 800.0 : 0.0);
      if (clk < best) {
        best = clk;
        p.tile = ts; p.splits = n; p.k_per = k_per; p.walk = s == 0 ? 1 : 0;
        p.gx = ceil_div(p.N, ts); p.units = tiles * n;
      }
    }
  }
  const bool ak = p.sak == 1, bk = p.sbk == 1 && p.sbn != 1;
  p.vec_a = es == 4 && ((uintptr_t)p.A & 15) == 0 && (ak ? p.sam : p.sak) % 4 == 0;
  p.vec_b = es == 4 && ((uintptr_t)p.Bm & 15) == 0 && (bk ? p.sbn : p.sbk) % 4 == 0;
  return best;
}
// The form of a contraction, and of a dW with the input gradient beside it (both in the same form: one launch has CTAs of one
// kind): the one with the least estimated time, for the rows that are expected (a same-sample dW; its grid covers p.M).
// The tensor-core form has to be ahead by 15 %, which is what the estimates are good for.
inline bool tc_wins(double cuda_cores, double tensor_cores) { return 1.15 * tensor_cores < cuda_cores; }
inline void plan_forms(GemmParams& p, int64_t rows, int es, int64_t k_step = 4, bool may_walk = true) {
  GemmParams c = p, t = p;
  const double est = plan_gemm(c, rows, es, k_step, may_walk);
  if (es == 4 && tc_wins(est, plan_gemm_tc(t, rows, k_step, false))) p = t;
  else plan_gemm(p, p.M, es, k_step, may_walk);
}
inline void plan_joint(GemmParams& w, GemmParams& g, int64_t rows, int es, int64_t k_step, bool may_walk) {
  GemmParams c = w, tw = w, tg = g;
  const double est = plan_gemm(c, rows, es, k_step, may_walk) + plan_gemm(g, g.M, es);
  if (es == 4 && tc_wins(est, plan_gemm_tc(tw, rows, k_step, true) + plan_gemm_tc(tg, g.M, 4, true))) {
    w = tw;
    g = tg;
  } else {
    plan_gemm(w, w.M, es, k_step, may_walk);
  }
}
// Waits for the kernel ahead and lets the next launch in, whatever the unit.
template <typename T, int EPI>
__device__ __forceinline__ void gemm_unit_partial(const GemmParams& p, int64_t unit, float* smem) {
  if (unit >= p.units) {
    begin_after_previous();
    return;
  }
  if constexpr (EPI != kEpiSparse) {
    if (p.walk) {
      begin_after_previous();
      if (p.tile == 32) gemm_walk<T, EPI, 32>(p, unit, smem); else gemm_walk<T, EPI, 64>(p, unit, smem);
      return;
    }
  }
  if (p.tile == 32) gemm_partial<T, EPI, 32>(p, (int)unit / p.splits, (int)unit % p.splits, smem);
  else gemm_partial<T, EPI, 64>(p, (int)unit / p.splits, (int)unit % p.splits, smem);
}
template <typename T, int EPI>
__device__ __forceinline__ void gemm_unit_finish(const GemmParams& p, int64_t unit, const float* smem) {
  if (unit >= p.units || p.walk) return;
  if (p.tile == 32) gemm_finish<T, EPI, 32>(p, (int)unit / p.splits, (int)unit % p.splits, smem);
  else gemm_finish<T, EPI, 64>(p, (int)unit / p.splits, (int)unit % p.splits, smem);
}

template <typename T, int EPI>
__global__ void __launch_bounds__(256, 2) gemm_kernel(const GemmParams p) {
  extern __shared__ __align__(16) float smem[];
  gemm_unit_partial<T, EPI>(p, blockIdx.x, smem);
  share_barrier();
  gemm_unit_finish<T, EPI>(p, blockIdx.x, smem);
  if (cluster_nctas() > 1) cluster_barrier();        // no CTA leaves while another reads its partial tile
}

// More CTAs than the chip holds at once (two per SM): the next launch is let in by each CTA's end, not by its beginning.  Its
// waiting CTAs in the slots beside the last wave cost that wave more than the gap between the launches (bf16 2000 x
// 1001 x 777 forward 177 against 156 us, input gradient of 2049^3 743 against 722).
template <typename T, int EPI>
__global__ void __launch_bounds__(256) gemm_walk_kernel(const GemmParams p) {
  wait_for_previous();
  const bool waves = gridDim.x > 2 * 148;
  if (!waves) let_next_start();
  extern __shared__ __align__(16) float smem[];
  if (p.tile == 32) gemm_walk<T, EPI, 32>(p, blockIdx.x, smem); else gemm_walk<T, EPI, 64>(p, blockIdx.x, smem);
  if (waves) let_next_start();
}

template <int EPI>
int launch_planned(int dtype, const GemmParams& p, cudaStream_t s) {
  if (p.units > 0x7fffffff) return RAD_EINVAL;
  if (p.tc) return launch_gemm_tc(EPI, p, s);
  count_launch();
  if constexpr (EPI != kEpiSparse) {
    if (p.walk) {
      const dim3 grid((unsigned)p.units);
      const size_t smem = (size_t)walk_smem_bytes(p.tile);
      return dtype == RAD_BF16 ? launch_kernel(gemm_walk_kernel<bf16, EPI>, grid, 256, smem, s, p)
                               : launch_kernel(gemm_walk_kernel<float, EPI>, grid, 256, smem, s, p);
    }
  }
  if (dtype == RAD_BF16) {
    static std::atomic<uint64_t> ready{0};
    if (!allow_smem(gemm_kernel<bf16, EPI>, kGemmSmemBytes, ready)) return RAD_ECUDA;
    return launch_with_cluster(gemm_kernel<bf16, EPI>, dim3((unsigned)p.units), 256, (size_t)gemm_smem_bytes(p.tile), dim3(p.splits), s, p);
  }
  static std::atomic<uint64_t> ready{0};
  if (!allow_smem(gemm_kernel<float, EPI>, kGemmSmemBytes, ready)) return RAD_ECUDA;
  return launch_with_cluster(gemm_kernel<float, EPI>, dim3((unsigned)p.units), 256, (size_t)gemm_smem_bytes(p.tile), dim3(p.splits), s, p);
}

template <int EPI>
int launch_gemm(int dtype, const GemmParams& p0, int64_t rows, cudaStream_t s) {
  GemmParams p = p0;
  plan_forms(p, rows, dtype == RAD_BF16 ? 2 : 4);
  return launch_planned<EPI>(dtype, p, s);
}

// relubits[b, w] = bits of (X[b, 32w..] > 0)
template <typename T>
__global__ void __launch_bounds__(256) relu_bits_rows_kernel(const T* X, int64_t ld, int64_t B, int64_t H,
                                                             int64_t w32, uint32_t* out) {
  begin_after_previous();
  const int64_t n = B * w32;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = i / w32, w = i % w32;
    const T* rowp = X + b * ld + w * 32;
    const int nv = (int)min((int64_t)32, H - w * 32);
    uint32_t m = 0;
    for (int c = 0; c < nv; ++c) m |= (to_float(rowp[c]) > 0.0f ? 1u : 0u) << c;
    out[i] = m;
  }
}

// dW of a layer and the gradient of its input in one launch: both read the same dZ and neither reads the
// other's result, so the first `dw_blocks` CTAs are those of the weight gradient in a launch of its own and the rest
// those of the input gradient, each doing exactly what it does there (the nets that run on CUDA cores are bound by
// their launch count).  `dw_blocks` is a multiple of the cluster size.
template <typename T>
__global__ void __launch_bounds__(256, 2) dw_dx_kernel(const GemmParams w, const GemmParams g, int dw_blocks) {
  extern __shared__ __align__(16) float smem[];
  const int b = (int)blockIdx.x, gu = b - dw_blocks;
  if (b < dw_blocks) gemm_unit_partial<T, kEpiSparse>(w, b, smem);
  else gemm_unit_partial<T, kEpiInputGrad>(g, gu, smem);
  share_barrier();
  if (b < dw_blocks) gemm_unit_finish<T, kEpiSparse>(w, b, smem);
  else gemm_unit_finish<T, kEpiInputGrad>(g, gu, smem);
  if (cluster_nctas() > 1) cluster_barrier();
}

__global__ void zero_rows_kernel(float* dW, int64_t ldw, int64_t D, int64_t H) {
  begin_after_previous();
  const int64_t n = D * H;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    dW[(i / H) * ldw + (i % H)] = 0.0f;
}

// ---- column sums (bias gradient) -----------------------------------------------------------------
// A CTA owns CL x V neighbouring columns (one 128-byte line where the matrix is wide) and a slab of rows: 256 / CL
// row lanes, each with V columns in registers and 16-byte loads where the layout allows them.  The lanes of a
// column are added by shuffles, the eight warps in shared memory, the CTAs of a cluster (its slabs of rows) by
// distributed shared memory: every sum in a fixed order, one launch.
// Bound by the latency of the loads in flight, so what matters is how many CTAs share the rows: with one CTA per
// 128 rows x 2048 columns (the form before) a 4096 x 2048 bf16 matrix (16.8 MB) took 56 + 5 us on 32 CTAs whose
// threads walked 128 rows each; here it is 256 CTAs of 16 rows per thread.
constexpr int kColMaxCluster = 8;          // portable cluster size
// From here on DRAM is what bounds the sum, and 512 bytes of a row per CTA read better than 128: 65536 x 8192 bf16
// 186 us (5.8 TB/s) against 216 us with clusters on 128-byte columns and 200 us before; 16384 x 4096 (134 MB), which
// L2 still helps, 33 against 30 us, so the line lies above it.
constexpr int64_t kColBigBytes = 256ll << 20;
constexpr int64_t kColTallRows = 128;      // rows of a thread above which one cluster along the rows is too few CTAs
template <typename T, int V>
__device__ __forceinline__ void colsum_load(const T* p, float (&v)[V]) {
  if constexpr (V == 1) {
    v[0] = to_float(*p);
  } else if constexpr (sizeof(T) == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  } else {
    const uint4 x = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[2 * i] = __uint_as_float(w[i] << 16);
      v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
}
// grid (column blocks, CTAs along the rows); the latter is the cluster size where `out` is the result itself, and
// the number of partial rows (cluster of one) where a second launch adds them
template <typename T, int V>
__global__ void __launch_bounds__(256) colsum_kernel(const T* dZ, int64_t ldz, int64_t B, int64_t H, int log_cl,
                                                     int64_t rows_per_cta, float* out, bool beside) {
  if (!beside) wait_for_previous();
  let_next_start();
  __shared__ float s_warp[8][32 * V];
  __shared__ float s_cta[32 * V];
  const int CL = 1 << log_cl, RL = 256 >> log_cl, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = tid & (CL - 1), r = tid >> log_cl;
  const int64_t h = ((int64_t)blockIdx.x * CL + c) * V;
  const int64_t b0 = (int64_t)blockIdx.y * rows_per_cta, b1 = min(B, b0 + rows_per_cta);
  float s[V] = {};
  if (h < H) {
    const T* p = dZ + h;
#pragma unroll 8
    for (int64_t b = b0 + r; b < b1; b += RL) {
      float v[V];
      colsum_load<T, V>(p + b * ldz, v);
#pragma unroll
      for (int i = 0; i < V; ++i) s[i] += v[i];
    }
  }
  for (int o = CL; o < 32; o <<= 1) {
#pragma unroll
    for (int i = 0; i < V; ++i) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
  }
  if (lane < CL) {
#pragma unroll
    for (int i = 0; i < V; ++i) s_warp[warp][lane * V + i] = s[i];
  }
  __syncthreads();
  const bool clustered = cluster_nctas() > 1;
  const int64_t hc = (int64_t)blockIdx.x * CL * V + tid;       // the column this thread finishes
  if (tid < CL * V) {
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += s_warp[w][tid];
    if (clustered) s_cta[tid] = t;
    else if (hc < H) out[(int64_t)blockIdx.y * H + hc] = t;
  }
  if (clustered) {
    cluster_barrier();
    if (blockIdx.y == 0 && tid < CL * V && hc < H) {
      float t = 0.0f;
      for (int q = 0; q < (int)gridDim.y; ++q) t += ld_cluster_f32(&s_cta[tid], (uint32_t)q);
      out[hc] = t;
    }
    cluster_barrier();                     // no CTA leaves while another reads its sums
  }
  if (beside && tid == 0) wait_for_previous();
}

template <typename T, int V>
int launch_colsum(const T* dZ, int64_t ldz, int64_t B, int64_t H, int log_cl, int ny, bool clustered, float* out, cudaStream_t s, bool beside = false) {
  const int64_t colblocks = ceil_div(H, (int64_t)V << log_cl);
  count_launch();
  return launch_with_cluster(colsum_kernel<T, V>, dim3((unsigned)colblocks, (unsigned)ny), 256, 0, clustered ? dim3(1, (unsigned)ny) : dim3(1),
                             s, dZ, ldz, B, H, log_cl, ceil_div(B, (int64_t)ny), out, beside);
}

// Column lanes of a CTA: eight 16-byte vectors make a 128-byte line; a narrow matrix gets the power of two that
// holds its columns, so that the other threads are row lanes.
template <typename T, int V>
int column_sums_of(const T* dZ, int64_t ldz, int64_t B, int64_t H, float* out, float* partial, int64_t max_slabs, cudaStream_t s, bool beside = false) {
  int log_cl = 0;
  const int64_t vecs = ceil_div(H, (int64_t)V);
  const bool big = V > 1 && vecs >= 32 && B * H * (int64_t)sizeof(T) >= kColBigBytes && max_slabs > kColMaxCluster;
  while ((1 << log_cl) < vecs && log_cl < (V > 1 && !big ? 3 : 5)) ++log_cl;
  const int64_t RL = 256 >> log_cl, colblocks = ceil_div(vecs, (int64_t)1 << log_cl);
  // one launch: enough CTAs per column block that a thread adds about four rows, at most a cluster
  int ny = 1;
  while (ny < kColMaxCluster && B > 4 * RL * ny) ny *= 2;
  // Two launches where a cluster per column block would leave most SMs idle and its threads with a long walk
  // (a convolution's bias gradient: B H W rows of 16 to 64 channels; 4.2 M x 16 bf16 took 75 + 19 us, the second
  // figure one CTA adding 296 partial rows one by one): first one partial row per slab, then the cluster form on those.
  // `tall`: so many rows that a thread of a cluster would add more than 128 of them one after the other, however many
  // column blocks there are; CTAs in whole waves of 1184 (eight per SM), at least sixteen slabs.  65536 x 601 float32 86 us
  // in one launch, 38 in two; bf16 80 and 31; 20000 x 5001 float32 93 and 75; 8192 x 601 (128 rows) 9.2 and 11.5.
  const bool tall = ny == kColMaxCluster && B > kColTallRows * RL * ny && max_slabs > kColMaxCluster;
  // (bf16 from twelve rows a thread on: 8192 x 64 5.5 us in one launch, 3.9 in two, 8192 x 256 5.7 and 4.2, 4096 x 256 4.0 and 3.6, 2100 x
  // 256 3.2 and 3.5; float32 8192 x 512 4.4 and 5.1)
  const bool narrow = ny == kColMaxCluster && colblocks * ny < 148 && B > (V == 8 ? 12 : 32) * RL * ny && max_slabs > kColMaxCluster;
  if (big || tall || narrow) {
    int64_t slabs = std::max<int64_t>(kColMaxCluster, (big ? 1184 : 592) / colblocks);
    if (tall && !big && !narrow)
      for (int64_t ctas = 1184; (slabs = ctas / colblocks) < 16; ctas += 1184) {}
    slabs = std::min(max_slabs, slabs);
    const int rc = launch_colsum<T, V>(dZ, ldz, B, H, log_cl, (int)slabs, false, partial, s);
    if (rc != RAD_OK) return rc;
    const bool vec = H % 4 == 0 && ((uintptr_t)partial & 15) == 0;
    return vec ? column_sums_of<float, 4>(partial, H, slabs, H, out, nullptr, 0, s)
               : column_sums_of<float, 1>(partial, H, slabs, H, out, nullptr, 0, s);
  }
  return launch_colsum<T, V>(dZ, ldz, B, H, log_cl, ny, true, out, s, beside);
}

}  // namespace

// The same for a same-sample store (Sec. 4.3): the first CTAs scatter A_c^T dZ into the kept rows of dW (and
// leave the bias gradient), the next ones make the input gradient, the last ones write zeros to the rows of dW
// whose column was not kept (bit d of keep_cols clear), which the scatter never touches.
// The parts begin at multiples of the cluster size.
template <typename T>
__global__ void __launch_bounds__(256, 2) same_dw_dx_kernel(const GemmParams w, const GemmParams g, int dw_blocks, int dx_blocks,
                                                            const uint32_t* keep_cols, int64_t D, int64_t H) {
  extern __shared__ __align__(16) float smem[];
  const int b = (int)blockIdx.x;
  if (b < dw_blocks) {
    gemm_unit_partial<T, kEpiScatterRows>(w, b, smem);
  } else if (b < dw_blocks + dx_blocks) {
    gemm_unit_partial<T, kEpiInputGrad>(g, b - dw_blocks, smem);
  } else {
    begin_after_previous();
    const int nz = (int)gridDim.x - dw_blocks - dx_blocks;
    for (int64_t d = b - dw_blocks - dx_blocks; d < D; d += nz) {
      if ((keep_cols[d >> 5] >> (d & 31)) & 1u) continue;
      for (int64_t h = threadIdx.x; h < H; h += 256) w.out_f32[d * w.ld_f32 + h] = 0.0f;
    }
  }
  share_barrier();
  if (b < dw_blocks) gemm_unit_finish<T, kEpiScatterRows>(w, b, smem);
  else if (b < dw_blocks + dx_blocks) gemm_unit_finish<T, kEpiInputGrad>(g, b - dw_blocks, smem);
  if (cluster_nctas() > 1) cluster_barrier();
}

int simt_forward(int dtype, int act, int64_t B, int64_t D, int64_t H, const void* A, int64_t lda,
                 const void* W, int64_t ldw, const float* bias, void* out_act, int64_t ld_act,
                 float* out_z, int64_t ld_z, void* out_zlow, int64_t ld_zlow, uint32_t* relubits,
                 int32_t* dev_status, cudaStream_t s) {
  GemmParams p = {};
  p.dev_status = dev_status;
  p.A = A; p.sam = lda; p.sak = 1;
  p.Bm = W; p.sbk = ldw; p.sbn = 1;
  p.M = B; p.N = H; p.K = D;
  p.bias = bias; p.act = act;
  p.out_act = out_act; p.ld_act = ld_act; p.out_z = out_z; p.ld_z = ld_z;
  p.out_zlow = out_zlow; p.ld_zlow = ld_zlow;
  int rc = launch_gemm<kEpiForward>(dtype, p, B, s);
  if (rc != RAD_OK) return rc;
  if (relubits != nullptr) {
    if (out_act == nullptr) return RAD_EINVAL;
    const int64_t w32 = ceil_div(H, 32), n = B * w32;
    const int g = (int)std::min<int64_t>(ceil_div(n, 256), 148 * 16);
    count_launch();
    if (dtype == RAD_BF16)
      RAD_TRY(launch_kernel(relu_bits_rows_kernel<bf16>, g, 256, 0, s, static_cast<const bf16*>(out_act), ld_act, B, H, w32, relubits));
    else
      RAD_TRY(launch_kernel(relu_bits_rows_kernel<float>, g, 256, 0, s, static_cast<const float*>(out_act), ld_act, B, H, w32, relubits));
  }
  return RAD_OK;
}

namespace {
GemmParams input_grad_params(int64_t B, int64_t D, int64_t H, const void* dZ, int64_t ldz, const SimtInputGrad& ig, int32_t* dev_status) {
  GemmParams p = {};
  p.dev_status = dev_status;
  p.A = dZ; p.sam = ldz; p.sak = 1;          // (b, h)
  p.Bm = ig.W; p.sbk = 1; p.sbn = ig.ldw;    // Bm(h, d) = W[d, h]
  p.M = B; p.N = D; p.K = H;
  p.relubits = ig.relubits_prev; p.w32 = ceil_div(D, 32);
  p.z_prev = ig.z_prev; p.ld_zprev = ig.ld_zprev;
  p.out_low = ig.dZ_prev; p.ld_low = ig.ldp;
  return p;
}
}  // namespace

int simt_input_grad(int dtype, int64_t B, int64_t D, int64_t H, const void* dZ, int64_t ldz,
                    const void* W, int64_t ldw, const uint32_t* relubits_prev, const void* z_prev,
                    int64_t ld_zprev, void* dZ_prev, int64_t ldp, int32_t* dev_status, cudaStream_t s) {
  const SimtInputGrad ig = {W, ldw, relubits_prev, z_prev, ld_zprev, dZ_prev, ldp};
  return launch_gemm<kEpiInputGrad>(dtype, input_grad_params(B, D, H, dZ, ldz, ig, dev_status), B, s);
}

int simt_weight_grad(const rad_store* st, const void* dZ, int64_t ldz, int64_t H, float* dW,
                     int64_t ldw, int32_t* dev_status, cudaStream_t s, float* db, bool* db_written,
                     const SimtInputGrad* ig, bool* ig_done) {
  if (db_written != nullptr) *db_written = false;
  if (ig_done != nullptr) *ig_done = false;
  if (st->variant == RAD_SAME_SAMPLE) {
    GemmParams p = {};
    p.dev_status = dev_status;
    p.A = st->values; p.sam = 1; p.sak = st->values_ld;     // A(j, b) = values[b, j]
    p.Bm = dZ; p.sbk = ldz; p.sbn = 1;
    p.M = min(st->values_ld, st->D); p.N = H; p.K = st->B;
    p.M_dev = st->nnz;
    p.row_idx = st->offsets; p.out_f32 = dW; p.ld_f32 = ldw;
    p.db = db;
    if (db_written != nullptr) *db_written = db != nullptr;
    const int es = st->dtype == RAD_BF16 ? 2 : 4;
    const int64_t rows = std::min(p.M, (int64_t)(1.05 * st->p * (double)st->D) + 16);
    if (st->keepbits != nullptr) {
      // one launch: scatter, zeros for the rows not kept and, where asked for, the input gradient
      const bool with_dx = ig != nullptr && ig_done != nullptr;
      GemmParams g = with_dx ? input_grad_params(st->B, st->D, H, dZ, ldz, *ig, dev_status) : GemmParams{};
      if (with_dx) plan_joint(p, g, rows, es, 4, true); else plan_forms(p, rows, es);
      const int64_t cluster = std::max(p.splits, with_dx ? g.splits : 1);
      const int64_t dw_blocks = round_up(p.units, cluster), dx_blocks = with_dx ? round_up(g.units, cluster) : 0;
      // zeros: two CTAs an SM where these fit beside the others, else the SMs the others leave (a tensor-core CTA has one)
      const int64_t rest = kNumSms - (dw_blocks + dx_blocks) % kNumSms;
      const int64_t nz = round_up(std::min<int64_t>(st->D, p.tc ? std::max<int64_t>(rest, 32) : 148 * 2), cluster);
      if (dw_blocks + dx_blocks + nz <= 0x7fffffff) {
        static std::atomic<uint64_t> ready_b{0}, ready_f{0};
        const dim3 grid((unsigned)(dw_blocks + dx_blocks + nz)), cl((unsigned)cluster);
        if (with_dx) *ig_done = true;
        if (p.tc)
          return launch_dw_dx_tc(kEpiScatterRows, p, with_dx ? &g : nullptr, dw_blocks, dx_blocks, nz, cluster,
                                 (const uint32_t*)st->keepbits, st->D, H, s);
        count_launch();
        if (st->dtype == RAD_BF16)
          return !allow_smem(same_dw_dx_kernel<bf16>, kGemmSmemBytes, ready_b) ? RAD_ECUDA
                 : launch_with_cluster(same_dw_dx_kernel<bf16>, grid, 256, kGemmSmemBytes, cl, s, p, g, (int)dw_blocks, (int)dx_blocks,
                                       (const uint32_t*)st->keepbits, st->D, H);
        return !allow_smem(same_dw_dx_kernel<float>, kGemmSmemBytes, ready_f) ? RAD_ECUDA
               : launch_with_cluster(same_dw_dx_kernel<float>, grid, 256, kGemmSmemBytes, cl, s, p, g, (int)dw_blocks, (int)dx_blocks,
                                     (const uint32_t*)st->keepbits, st->D, H);
      }
    }
    const int g = (int)std::min<int64_t>(ceil_div(st->D * H, 256), 148 * 16);
    count_launch();
    RAD_TRY(launch_kernel(zero_rows_kernel, g, 256, 0, s, dW, ldw, st->D, H));
    return launch_gemm<kEpiScatterRows>(st->dtype, p, rows, s);
  }
  const bool low = st->dtype == RAD_BF16;
  GemmParams p = {};
  p.dev_status = dev_status;
  p.A = st->values; p.keepbits = st->keepbits; p.offsets = st->offsets; p.capacity = st->values_capacity;
  p.ncb = (int32_t)ceil_div(st->D, kTileCols);
  p.Bm = dZ; p.sbk = ldz; p.sbn = 1;
  p.M = st->D; p.N = H; p.K = st->B;
  p.out_f32 = dW; p.ld_f32 = ldw;
  p.db = db;
  if (db_written != nullptr) *db_written = db != nullptr;
  const int es = low ? 2 : 4;
  if (ig != nullptr && ig_done != nullptr) {
    GemmParams g = input_grad_params(st->B, st->D, H, dZ, ldz, *ig, dev_status);
    plan_joint(p, g, p.M, es, kTileRows, false);
    const int64_t cluster = std::max(p.splits, g.splits), dw_blocks = round_up(p.units, cluster);
    const int64_t all = dw_blocks + round_up(g.units, cluster);
    if (all <= 0x7fffffff) {
      static std::atomic<uint64_t> ready_b{0}, ready_f{0};
      const size_t smem = (size_t)std::max(gemm_smem_bytes(g.tile), gemm_smem_bytes(p.tile));
      const dim3 grid((unsigned)all), cl((unsigned)cluster);
      *ig_done = true;
      if (p.tc) return launch_dw_dx_tc(kEpiSparse, p, &g, dw_blocks, all - dw_blocks, 0, cluster, nullptr, 0, 0, s);
      count_launch();
      if (low)
        return !allow_smem(dw_dx_kernel<bf16>, kGemmSmemBytes, ready_b) ? RAD_ECUDA
               : launch_with_cluster(dw_dx_kernel<bf16>, grid, 256, smem, cl, s, p, g, (int)dw_blocks);
      return !allow_smem(dw_dx_kernel<float>, kGemmSmemBytes, ready_f) ? RAD_ECUDA
             : launch_with_cluster(dw_dx_kernel<float>, grid, 256, smem, cl, s, p, g, (int)dw_blocks);
    }
  }
  plan_forms(p, p.M, es, kTileRows, false);
  return launch_planned<kEpiSparse>(st->dtype, p, s);
}

constexpr int kColChunkRows = 128;         // rows of dZ per partial row of the workspace
int64_t column_sums_workspace(int64_t B, int64_t H) {
  return round_up(ceil_div(B, kColChunkRows) * H * 4, 256);
}

int column_sums(int dtype, int64_t B, int64_t H, const void* dZ, int64_t ldz, float* db, void* workspace,
                int64_t workspace_bytes, cudaStream_t s, bool beside) {
  if (workspace == nullptr || workspace_bytes < column_sums_workspace(B, H)) return RAD_EWORKSPACE;
  float* partial = static_cast<float*>(workspace);
  const int64_t slabs = ceil_div(B, kColChunkRows);          // partial rows the workspace holds
  const bool aligned = ((uintptr_t)dZ & 15) == 0;
  if (dtype == RAD_BF16) {
    const bf16* z = static_cast<const bf16*>(dZ);
    return aligned && H % 8 == 0 && ldz % 8 == 0 ? column_sums_of<bf16, 8>(z, ldz, B, H, db, partial, slabs, s, beside)
                                                 : column_sums_of<bf16, 1>(z, ldz, B, H, db, partial, slabs, s, beside);
  }
  const float* z = static_cast<const float*>(dZ);
  return aligned && H % 4 == 0 && ldz % 4 == 0 ? column_sums_of<float, 4>(z, ldz, B, H, db, partial, slabs, s, beside)
                                               : column_sums_of<float, 1>(z, ldz, B, H, db, partial, slabs, s, beside);
}

}  // namespace rad
