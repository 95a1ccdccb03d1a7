// Index part of a different-sample store from the key alone (Sec. 3.2: the random P is independent of the
// data; Sec. 4.2: it is drawn per layer input).  The keep decision of entry (b, d) depends on (seed, layer,
// step, b, d) only, so keep bits, row offsets, tile offsets and the kept count can be produced without
// reading the layer input, before that input exists.  The forward GEMM of the layer that produces the input
// then drops the kept values into place from its epilogue (tc.cu), and a caller learns the exact size of a
// store before it allocates `values`.
//
// The index parts of all layers of a net are drawn in one go (a net's layers share seed, step and keep probability).
//
//   store_index_small_kernel  layers of few tiles: one launch, a cluster of eight CTAs per layer, which hand their kept
//                             counts on through distributed shared memory
//   store_index_kernel        one tile (64 x 128 entries) per warp and turn: draw and write the keep-bit words,
//                             in-tile row offsets from warp scans, exact kept count of the tile into offsets[tile]
//   offsets_scan_kernel       one CTA per layer turns the counts into padded exclusive prefixes in place and writes nnz
//
// Layout and bits are those of the one-pass store kernels.
#include <algorithm>

#include "common.cuh"

namespace rad {
namespace {

struct IndexLayer {
  uint32_t rows, cols, ncb, ntiles;
  uint32_t tile0;       // tiles of the layers before it
  uint32_t c2;
  uint32_t* keepbits;
  uint32_t* offsets;
  int64_t* nnz;
  int64_t capacity;     // elements of `values` the caller holds; < 0: not checked
};
constexpr int kIndexLayers = 16;   // layers of one launch
template <int kLayers>
struct IndexParams {
  IndexLayer layer[kLayers];
  int32_t nlayers;
  uint32_t ntiles;      // of all of them
  KeepThreshold T;
  uint32_t c3;
  int32_t* dev_status;
};

// One tile by one warp, no CTA-wide step: lane l draws words l, l + 32, ... of the tile (word t = row t / 4, columns
// 32 (t % 4) ..), so a warp's stores are contiguous and a warp scan per turn, carried over the eight turns, gives every
// row its offset in (row, column) order.  `tw`: the tile's words, in `keepbits` or in shared memory.  Returns the tile's kept count.
__device__ __forceinline__ uint32_t index_tile(const IndexLayer& L, uint32_t tile, const KeepThreshold& T, uint32_t c3, const PhiloxKeys& ks,
                                               int lane, uint32_t* tw) {
  const uint32_t slab = tile / L.ncb, cb = tile - slab * L.ncb;
  const int w = lane & 3;
  const uint32_t col0 = cb * kTileCols + 32u * w;
  uint32_t base = 0;
#pragma unroll 2
  for (int i = 0; i < kBitWords / 32; ++i) {
    const int r = i * 8 + (lane >> 2);
    const uint32_t row = slab * kTileRows + r;
    uint32_t m = 0;
    if (row < L.rows && col0 < L.cols) {
      m = philox_keep32(col0 >> 5, row, L.c2, c3, ks, T);
      const uint32_t nv = L.cols - col0;
      if (nv < 32) m &= (1u << nv) - 1u;
    }
    tw[i * 32 + lane] = m;
    const uint32_t c = __popc(m);
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t n = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += n;
    }
    if (w == 0) reinterpret_cast<uint16_t*>(tw + kBitWords)[r] = (uint16_t)(base + incl - c);
    base += __shfl_sync(0xffffffffu, incl, 31);
  }
  return base;
}
__device__ __forceinline__ uint32_t* tile_words(const IndexLayer& L, uint32_t tile) { return L.keepbits + (int64_t)tile * kTileWords; }
// A tile that was drawn into shared memory to its place, by its warp.
__device__ __forceinline__ void place_tile(const IndexLayer& L, uint32_t tile, const uint32_t* words, int lane) {
  uint32_t* tw = tile_words(L, tile);
  __syncwarp();
  if (((uintptr_t)tw & 15) == 0) {
    for (int i = lane; i < kTileWords / 4; i += 32) reinterpret_cast<uint4*>(tw)[i] = reinterpret_cast<const uint4*>(words)[i];
  } else {
    for (int i = lane; i < kTileWords; i += 32) tw[i] = words[i];
  }
}
__device__ __forceinline__ uint32_t padded_count(uint32_t c) { return (c + kValueAlign - 1) / kValueAlign * kValueAlign; }
__device__ __forceinline__ void write_totals(const IndexLayer& L, uint32_t padded, uint32_t exact, int32_t* dev_status) {
  L.offsets[L.ntiles] = padded;
  L.nnz[0] = (int64_t)exact;
  L.nnz[1] = (int64_t)padded;
  if (L.capacity >= 0 && (int64_t)padded > L.capacity) raise_status(dev_status, RAD_DEV_ECAPACITY);
}

constexpr int kIndexWarps = 16;
// (One layer has a form of its own: fewer registers, 65536 tiles 160 us instead of 163.)
// ahead: a tile per warp at most, drawn into the shared memory that spreads the CTAs before the kernel ahead has ended: the key is
// all it takes.
template <int kLayers>
__global__ void __launch_bounds__(32 * kIndexWarps) store_index_kernel(const __grid_constant__ IndexParams<kLayers> p, const PhiloxKeys ks, int ahead) {
  const int lane = threadIdx.x & 31;
  if (ahead) {
    extern __shared__ __align__(16) uint32_t s_tiles[];
    const uint32_t t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    uint32_t* words = s_tiles + (threadIdx.x >> 5) * kTileWords;
    int l = 0;
    if (kLayers > 1)
      while (l + 1 < p.nlayers && t >= p.layer[l + 1].tile0) ++l;
    const IndexLayer layer = p.layer[l];
    uint32_t count = 0;
    if (t < p.ntiles) count = index_tile(layer, t - layer.tile0, p.T, p.c3, ks, lane, words);
    begin_after_previous();
    if (t < p.ntiles) {
      place_tile(layer, t - layer.tile0, words, lane);
      if (lane == 0) layer.offsets[t - layer.tile0] = count;
    }
    return;
  }
  wait_for_previous();
  const uint32_t warps = blockDim.x >> 5, warp0 = blockIdx.x * warps + (threadIdx.x >> 5), nwarps = gridDim.x * warps;
  int l = 0;
  IndexLayer layer = p.layer[0];                    // in registers: out of the parameters by a variable index, every use would be a load
  for (uint32_t t = warp0; t < p.ntiles; t += nwarps) {
    if ((uint64_t)t + nwarps >= p.ntiles) let_next_start();
    if (kLayers > 1)
      while (l + 1 < p.nlayers && t >= p.layer[l + 1].tile0) layer = p.layer[++l];
    const uint32_t tile = t - layer.tile0;
    const uint32_t count = index_tile(layer, tile, p.T, p.c3, ks, lane, tile_words(layer, tile));
    if (lane == 0) layer.offsets[tile] = count;
  }
}

// Layers of at most kSmallIndexTiles tiles: cluster l (eight CTAs) makes layer l, CTA r of it a run of its tiles.  What
// bounds a small index is launches, not the draw: drawn and scanned in two launches per layer, the layers of a
// 640-520-392-200 net at batch 328 took 20 us of its step, in one launch for all of them 6.  An SM draws a tile in 0.26 us (three generator calls per word, 3 G calls/s), so with
// more than twelve tiles a CTA the two launches of the general form, on all SMs, are faster.
constexpr int kSmallIndexCtas = 8, kSmallIndexTiles = 12 * kSmallIndexCtas;
// Everything but the writes is done before the kernel ahead has ended: the key is all it takes.
__global__ void __launch_bounds__(32 * kIndexWarps) store_index_small_kernel(const __grid_constant__ IndexParams<kIndexLayers> p, const PhiloxKeys ks) {
  cluster_started_arrive();                             // waited for behind the draw
  constexpr int kTiles = kSmallIndexTiles / kSmallIndexCtas;
  static_assert(kTiles <= kIndexWarps, "a tile per warp");
  __shared__ __align__(16) uint32_t s_words[kTiles][kTileWords];
  __shared__ uint32_t s_count[kTiles];
  __shared__ uint32_t s_padded[kSmallIndexCtas], s_exact[kSmallIndexCtas];      // of every CTA of the cluster
  const IndexLayer& L = p.layer[blockIdx.x / kSmallIndexCtas];
  const uint32_t rank = cluster_ctarank(), per = (L.ntiles + kSmallIndexCtas - 1) / kSmallIndexCtas;
  const uint32_t t0 = min(rank * per, L.ntiles), n = min(per, L.ntiles - t0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp < n) {
    const uint32_t count = index_tile(L, t0 + warp, p.T, p.c3, ks, lane, s_words[warp]);
    if (lane == 0) s_count[warp] = count;
  }
  __syncthreads();
  cluster_started_wait();                               // before the first write to a peer: a CTA without tiles is here at once
  if (tid < kSmallIndexCtas) {
    uint32_t padded = 0, exact = 0;
    for (uint32_t i = 0; i < n; ++i) {
      padded += padded_count(s_count[i]);
      exact += s_count[i];
    }
    st_cluster_u32(&s_padded[rank], (uint32_t)tid, padded);
    st_cluster_u32(&s_exact[rank], (uint32_t)tid, exact);
  }
  cluster_barrier();
  begin_after_previous();
  if (warp < n) place_tile(L, t0 + warp, s_words[warp], lane);
  if (tid == 0) {
    uint32_t at = 0, exact = 0, all = 0;
    for (uint32_t r = 0; r < kSmallIndexCtas; ++r) {
      if (r < rank) at += s_padded[r];
      all += s_padded[r];
      exact += s_exact[r];
    }
    for (uint32_t i = 0; i < n; ++i) {
      L.offsets[t0 + i] = at;
      at += padded_count(s_count[i]);
    }
    if (rank == 0) write_totals(L, all, exact, p.dev_status);
  }
}

// offsets[t] holds the exact kept count of tile t on entry and the first element of tile t in `values` on
// exit (every tile padded to a multiple of kValueAlign); offsets[ntiles] = elements used.  One CTA, 16384
// tiles per round; a thread takes 16 consecutive tiles (four 16-byte loads and stores where `offsets` is
// 16-byte aligned), adds them up locally, and one warp scan plus one pass over the warp sums places them.
constexpr int kScanPer = 16;
template <int kLayers>
__global__ void __launch_bounds__(1024) offsets_scan_kernel(const __grid_constant__ IndexParams<kLayers> p) {
  begin_after_previous();
  const IndexLayer L = p.layer[kLayers > 1 ? blockIdx.x : 0];
  uint32_t* offsets = L.offsets;
  const bool vec = ((uintptr_t)offsets & 15) == 0;
  __shared__ uint64_t s_warp[32];                   // padded sum in the high half, exact sum in the low half
  __shared__ uint64_t s_carry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_carry = 0;
  __syncthreads();
  const int64_t ntiles = L.ntiles;
  for (int64_t r0 = 0; r0 < ntiles; r0 += 1024 * kScanPer) {
    const int64_t t0 = r0 + (int64_t)tid * kScanPer;
    const bool whole = vec && t0 + kScanPer <= ntiles;
    uint32_t c[kScanPer];
    if (whole) {
#pragma unroll
      for (int i = 0; i < kScanPer; i += 4) {
        const uint4 q = *reinterpret_cast<const uint4*>(offsets + t0 + i);
        c[i] = q.x; c[i + 1] = q.y; c[i + 2] = q.z; c[i + 3] = q.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < kScanPer; ++i) c[i] = t0 + i < ntiles ? offsets[t0 + i] : 0u;
    }
    // a round holds at most 16384 * 8192 entries: 32 bits each for the padded and the exact sum
    uint64_t mine = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i)
      mine += ((uint64_t)((c[i] + kValueAlign - 1) / kValueAlign * kValueAlign) << 32) | c[i];
    uint64_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t n = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += n;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    const uint64_t carry = s_carry;
    uint64_t before = incl - mine, round_total = 0;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const uint64_t t = s_warp[i];
      if (i < warp) before += t;
      round_total += t;
    }
    uint32_t at = (uint32_t)((carry >> 32) + (before >> 32));     // the padded total stays below 2^32
    uint32_t o[kScanPer];
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
      o[i] = at;
      at += (c[i] + kValueAlign - 1) / kValueAlign * kValueAlign;
    }
    if (whole) {
#pragma unroll
      for (int i = 0; i < kScanPer; i += 4)
        *reinterpret_cast<uint4*>(offsets + t0 + i) = make_uint4(o[i], o[i + 1], o[i + 2], o[i + 3]);
    } else {
#pragma unroll
      for (int i = 0; i < kScanPer; ++i)
        if (t0 + i < ntiles) offsets[t0 + i] = o[i];
    }
    __syncthreads();                                // everyone has read the carry and the warp sums
    if (tid == 0) s_carry = carry + round_total;
    __syncthreads();
  }
  if (tid == 0) {
    const uint64_t total = s_carry;
    write_totals(L, (uint32_t)(total >> 32), (uint32_t)(total & 0xffffffffu), p.dev_status);
  }
}

}  // namespace

// Exact kept counts per tile in offsets[0 .. ntiles) -> padded exclusive prefixes, offsets[ntiles] and nnz.
int launch_offsets_scan(uint32_t* offsets, int64_t ntiles, int64_t* nnz, int64_t capacity, int32_t* dev_status,
                        cudaStream_t s) {
  IndexParams<1> p = {};
  p.nlayers = 1; p.dev_status = dev_status;
  p.layer[0].ntiles = (uint32_t)ntiles; p.layer[0].offsets = offsets; p.layer[0].nnz = nnz; p.layer[0].capacity = capacity;
  count_launch();
  return launch_kernel(offsets_scan_kernel<1>, 1, 1024, 0, s, p);
}

namespace {
// Up to kLayers layers of one seed, step and keep probability: the general form.
template <int kLayers>
int launch_index_tiles(const IndexParams<kLayers>& p, const PhiloxKeys& ks, cudaStream_t s) {
  // Tiles spread over all SMs: an SM draws one in 0.26 us, so 256 tiles are for 64 SMs and not for sixteen (7.7 us with the scan
  // instead of 10.6).  Up to sixteen tiles an SM one CTA of as many warps as that takes, at least four, and the shared memory
  // says so: started early beside a tensor-core kernel that leaves a few SMs idle, CTAs without that share those few (1024
  // tiles behind an input gradient on 128 of 148 SMs: 12.5 us, 6 otherwise).  More tiles: CTAs of four warps (8192 tiles 23.4 us,
  // 25.4 with five of eight an SM), and of eight where every warp has several (16384 tiles 41.1 us, 43.3 with four).
  static std::atomic<uint64_t> ready{0};
  if (!allow_smem(store_index_kernel<kLayers>, kSpreadSmemMax, ready)) return RAD_ECUDA;
  const int64_t per_sm = ceil_div(p.ntiles, kNumSms);
  const int warps = per_sm <= 4 ? 4 : per_sm <= 8 ? 8 : per_sm <= kIndexWarps ? kIndexWarps : per_sm <= 64 ? 4 : 8;
  const int64_t most = (per_sm <= kIndexWarps ? 1 : per_sm <= 64 ? 12 : 5) * kNumSms, ctas = std::min(ceil_div(p.ntiles, warps), most);
  count_launch();
  const size_t smem = spread_smem(ctas, 0);
  const int ahead = ctas * warps >= p.ntiles && smem >= (size_t)warps * kTileWords * 4 ? 1 : 0;
  RAD_TRY(launch_kernel(store_index_kernel<kLayers>, (unsigned)ctas, 32 * warps, smem, s, p, ks, ahead));
  count_launch();
  return launch_kernel(offsets_scan_kernel<kLayers>, p.nlayers, 1024, 0, s, p);
}
}  // namespace

// Index parts (keep bits, row offsets, tile offsets, nnz) of the different-sample Bernoulli stores of one net: one seed,
// step and keep probability.
int launch_store_indices(const rad_store* st, int n, bool check_capacity, int32_t* dev_status, cudaStream_t s) {
  const PhiloxKeys ks = philox_expand_key(st[0].seed);
  for (int first = 0; first < n; first += kIndexLayers) {
    IndexParams<kIndexLayers> p = {};
    p.nlayers = std::min(n - first, kIndexLayers);
    p.T = make_keep_threshold(keep_threshold_host(st[0].p));
    p.c3 = st[0].step;
    p.dev_status = dev_status;
    bool small = true;
    for (int l = 0; l < p.nlayers; ++l) {
      const rad_store& q = st[first + l];
      IndexLayer& L = p.layer[l];
      L.rows = (uint32_t)q.B; L.cols = (uint32_t)q.D;
      L.ncb = (uint32_t)ceil_div(q.D, kTileCols);
      L.ntiles = (uint32_t)ceil_div(q.B, kTileRows) * L.ncb;
      L.tile0 = p.ntiles;
      L.c2 = counter_word2(q.layer, RAD_DIFFERENT_SAMPLE);
      L.keepbits = q.keepbits; L.offsets = q.offsets; L.nnz = q.nnz;
      L.capacity = check_capacity ? q.values_capacity : -1;
      p.ntiles += L.ntiles;
      small = small && L.ntiles <= (uint32_t)kSmallIndexTiles;
    }
    if (small) {
      count_launch();
      RAD_TRY(launch_with_cluster(store_index_small_kernel, p.nlayers * kSmallIndexCtas, 32 * kIndexWarps, 0, dim3(kSmallIndexCtas, 1, 1),
                                  s, p, ks));
    } else if (p.nlayers == 1) {
      RAD_TRY(launch_index_tiles(IndexParams<1>{{p.layer[0]}, 1, p.ntiles, p.T, p.c3, p.dev_status}, ks, s));
    } else {
      RAD_TRY(launch_index_tiles(p, ks, s));
    }
  }
  return RAD_OK;
}

// Index part of one different-sample store.
int launch_store_index(const rad_store* st, bool check_capacity, int32_t* dev_status, cudaStream_t s) {
  if (st->law == RAD_LAW_FIXED) return launch_fixed_index(st, check_capacity, dev_status, s);
  return launch_store_indices(st, 1, check_capacity, dev_status, s);
}

}  // namespace rad

using namespace rad;

extern "C" int rad_store_index(const rad_store* st, int32_t* dev_status, void* stream) {
  if (st == nullptr || st->B <= 0 || st->D <= 0) return RAD_EINVAL;
  if (st->variant != RAD_DIFFERENT_SAMPLE || (st->law != RAD_LAW_BERNOULLI && st->law != RAD_LAW_FIXED)) return RAD_EUNSUPPORTED;
  if (st->keepbits == nullptr || st->offsets == nullptr || st->nnz == nullptr) return RAD_EINVAL;
  if (keep_threshold_host(st->p) == 0) return RAD_EINVAL;
  if ((double)st->B * (double)st->D >= 4294967296.0 * 0.75) return RAD_EINVAL;
  const int rc = check_device();
  if (rc != RAD_OK) return rc;
  return launch_store_index(st, st->values != nullptr, dev_status, static_cast<cudaStream_t>(stream));
}
