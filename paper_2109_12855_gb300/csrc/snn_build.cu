// snn_build.cu -- construction of the source-major connection store on the
// device (network construction is outside the paper's measurements, Section
// 2.2; the store layout follows its Section 3.1: source-specific target
// segments).
//
// Pipeline: (1) count out-degrees with one generator call per synapse,
// (2) the host turns them into row offsets, (3) scatter one 64-bit sort key
// per synapse into its row, (4) sort every row by key in shared memory
// (bitonic network; rows longer than the shared-memory capacity are sorted
// in a global scratch buffer), pack the records (regenerating the weight from
// the key's tie field) and write the row's target-tile index.
//
// Sort key, for target tiles of TW neurons (tile = target / TW, position in
// the tile lo = target - tile TW < 2^B with B = lo_bits):
//   tile (24 - B bits) | delay (8) | lo (B) | tie (32)
// so a row is ordered by (target tile, delay, target, tie), where tie is the
// draw index k (fixed in-degree rule) or the edge index.  Sorting by the full
// key makes the store independent of the scatter's atomic order.  Within a
// tile a row is sorted by (delay, target); the tile index tile_off[row][tau]
// is the offset (relative to the row) of the first record of tile tau, for
// tau = 0 .. n_tiles (the last entry is the row length).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "snn_internal.cuh"

namespace snn {
namespace {

struct TileGeom {
  uint32_t tw;  // targets per tile
  int lb;       // bits of the position within a tile
};

__device__ __forceinline__ uint64_t make_key(uint32_t d, uint32_t tgt,
                                             uint32_t tie, TileGeom g) {
  const uint32_t tile = tgt / g.tw, lo = tgt - tile * g.tw;
  return ((uint64_t)tile << (40 + g.lb)) | ((uint64_t)(d & 0xFFu) << (32 + g.lb)) |
         ((uint64_t)lo << 32) | tie;
}
__device__ __forceinline__ uint32_t key_target(uint64_t key, TileGeom g) {
  return (uint32_t)(key >> (40 + g.lb)) * g.tw +
         ((uint32_t)(key >> 32) & ((1u << g.lb) - 1u));
}
__device__ __forceinline__ uint32_t key_delay(uint64_t key, TileGeom g) {
  return (uint32_t)(key >> (32 + g.lb)) & 0xFFu;
}

__device__ __forceinline__ uint32_t fixed_source(const BuildFixed& b,
                                                 uint32_t k, uint32_t u) {
  return k < b.k_e ? scale_u32(u, b.n_e) : b.n_e + scale_u32(u, b.n_i);
}

// One block per local target (the draws use its global index); a grid
// smaller than the targets walks them in strides (a build confined to some
// SMs, see BuildShape).
__global__ void __launch_bounds__(1024) k_count_fixed(BuildFixed b, uint32_t* deg) {
  const uint32_t kk = b.k_e + b.k_i;
  for (uint32_t tgt = blockIdx.x; tgt < b.n_tgt; tgt += gridDim.x)
    for (uint32_t k = threadIdx.x; k < kk; k += blockDim.x) {
      U4 r = draw(b.seed, b.tgt0 + tgt, k, 0u);
      atomicAdd(&deg[fixed_source(b, k, r.x)], 1u);
    }
}

__global__ void __launch_bounds__(1024) k_scatter_fixed(BuildFixed b, const uint64_t* row_ptr,
                                uint32_t* cursor, uint64_t* keys, TileGeom g) {
  const uint32_t kk = b.k_e + b.k_i;
  const uint32_t span = (uint32_t)(b.d_hi - b.d_lo + 1);
  for (uint32_t tgt = blockIdx.x; tgt < b.n_tgt; tgt += gridDim.x)
    for (uint32_t k = threadIdx.x; k < kk; k += blockDim.x) {
      U4 r = draw(b.seed, b.tgt0 + tgt, k, 0u);
      uint32_t src = fixed_source(b, k, r.x);
      uint32_t d = (uint32_t)b.d_lo + scale_u32(r.y, span);
      uint32_t pos = atomicAdd(&cursor[src], 1u);
      keys[row_ptr[src] + pos] = make_key(d, tgt, k, g);
    }
}

// The same counts with each CTA's counters in its shared memory, for
// populations that fit there: CTA c draws for the targets [c per, (c + 1) per)
// and adds its counts once per source at the end.  One global atomic per
// synapse bounded the plain form (1.2e11/s): 30,011 neurons of in-degree 3,000,
// 0.78 -> 0.25 ms; 112,500 of 11,250, 7.1 -> 3.2 ms.  (A scatter that takes its
// places from such counters too was slower, 1.4 -> 3.3 ms: every row is then
// written at as many places at once as there are CTAs, more partly written
// sectors than L2 holds.)
// W16: counters in halves of a word (a CTA draws a source at most 65,535
// times: count_shared).
template <bool W16>
__global__ void __launch_bounds__(1024) k_count_shared(BuildFixed b, uint32_t n_src,
                                                       uint32_t per, uint32_t* deg) {
  extern __shared__ uint32_t sc[];
  const uint32_t kk = b.k_e + b.k_i;
  const uint32_t words = W16 ? (n_src + 1) / 2 : n_src;
  for (uint32_t k = threadIdx.x; k < words; k += blockDim.x) sc[k] = 0;
  __syncthreads();
  const uint32_t lo = blockIdx.x * per, hi = min(lo + per, b.n_tgt);
  for (uint32_t tgt = lo; tgt < hi; ++tgt)
    for (uint32_t k = threadIdx.x; k < kk; k += blockDim.x) {
      const U4 r = draw(b.seed, b.tgt0 + tgt, k, 0u);
      const uint32_t src = fixed_source(b, k, r.x);
      if (W16) atomicAdd(&sc[src >> 1], 1u << (16u * (src & 1u)));
      else atomicAdd(&sc[src], 1u);
    }
  __syncthreads();
  for (uint32_t k = threadIdx.x; k < n_src; k += blockDim.x) {
    const uint32_t x = W16 ? (sc[k >> 1] >> (16u * (k & 1u))) & 0xFFFFu : sc[k];
    if (x) atomicAdd(&deg[k], x);
  }
}

__global__ void k_count_edges(const uint32_t* src, uint64_t n, uint32_t* deg) {
  for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < n;
       e += (uint64_t)gridDim.x * blockDim.x)
    atomicAdd(&deg[src[e]], 1u);
}

__global__ void k_scatter_edges(const uint32_t* src, const uint32_t* tgt,
                                const uint8_t* delay, uint64_t n,
                                const uint64_t* row_ptr, uint32_t* cursor,
                                uint64_t* keys, TileGeom g) {
  for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < n;
       e += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t s = src[e];
    uint32_t pos = atomicAdd(&cursor[s], 1u);
    keys[row_ptr[s] + pos] = make_key(delay[e], tgt[e], (uint32_t)e, g);
  }
}

// Weight of a synapse, FP64: per-edge value, or the fixed rule's mean plus
// a Box-Muller normal from words 2 and 3 of the synapse's draw.
template <int WMODE>
__device__ double weight_of(const BuildFixed& b, const double* edge_w,
                            bool exc, uint32_t tgt, uint32_t tie) {
  if (WMODE == 1) return edge_w[tie];
  double mean = exc ? b.w_e : b.w_i, sd = exc ? b.sd_e : b.sd_i;
  double x = mean;
  if (sd != 0.0) {
    U4 r = draw(b.seed, b.tgt0 + tgt, tie, 0u);
    double u1 = ((double)r.z + 1.0) * 0x1p-32;
    double u2 = (double)r.w * 0x1p-32;
    double z = sqrt(-2.0 * log(u1)) * cos(2.0 * 3.14159265358979323846 * u2);
    x = mean + sd * z;
  }
  if (exc && b.clip_e && x < 0.0) x = 0.0;
  if (!exc && b.clip_i && x > 0.0) x = 0.0;
  return x;
}

// BF16 bits of a fixed-rule weight.  The rounding to 8 significant bits is
// decided from an FP32 evaluation of the same Box-Muller normal whenever the
// FP32 value's error bound lies inside one rounding interval, and only
// otherwise (about 0.2 % of the draws) from the FP64 evaluation: rounding is
// monotonic, so if both ends of [x - e, x + e] round to the same BF16 value,
// the FP64 value does too.  The result equals the FP64 path's, at a small
// fraction of its cost (FP64 arithmetic is a small share of this GPU's
// throughput).  Bound: with the CUDA math library's documented maximum
// errors (1 ulp for logf, log1pf and cospif; sqrtf correctly rounded) and
// the conversions of the draw words to float, |s| <= 6.67 and
// |dz| <= 14 2^-21 < 2^-16; the conversions of mean and sd and the final
// fused multiply-add add at most 2^-23 (|mean| + 7 |sd|).
__device__ uint16_t bf16_weight_bits(const BuildFixed& b, bool exc,
                                     uint32_t tgt, uint32_t tie) {
  const double mean = exc ? b.w_e : b.w_i, sd = exc ? b.sd_e : b.sd_i;
  const bool clip_lo = exc && b.clip_e, clip_hi = !exc && b.clip_i;
  if (sd == 0.0) {
    double x = mean;
    if (clip_lo && x < 0.0) x = 0.0;
    if (clip_hi && x > 0.0) x = 0.0;
    return bf16_bits_rne(x);
  }
  const U4 r = draw(b.seed, b.tgt0 + tgt, tie, 0u);
  // ln u1 for u1 = (z + 1) 2^-32: directly below 1/2; above it as
  // log1p(u1 - 1) with u1 - 1 = -(2^32 - 1 - z) 2^-32 (no cancellation)
  const float ln = r.z < 0x7FFFFFFFu ? logf(((float)r.z + 1.0f) * 0x1p-32f)
                                     : log1pf(-(float)(~r.z) * 0x1p-32f);
  const float sv = sqrtf(-2.0f * ln);
  const float cv = cospif(2.0f * ((float)r.w * 0x1p-32f));
  const float sdf = (float)sd, meanf = (float)mean;
  const float xf = fmaf(sdf, sv * cv, meanf);
  const float e = fabsf(sdf) * 0x1p-16f +
                  (fabsf(meanf) + 7.0f * fabsf(sdf)) * 0x1p-20f;
  float lo = __fsub_rd(xf, e), hi = __fadd_ru(xf, e);
  if (clip_lo) {
    lo = fmaxf(lo, 0.0f);
    hi = fmaxf(hi, 0.0f);
  }
  if (clip_hi) {
    lo = fminf(lo, 0.0f);
    hi = fminf(hi, 0.0f);
  }
  const uint16_t a = bf16_bits_rne((double)lo);
  if (a == bf16_bits_rne((double)hi)) return a;
  return bf16_bits_rne(weight_of<0>(b, nullptr, exc, tgt, tie));
}

// Stored form of a fixed-rule or edge weight: the float, or the bfloat16 bits.
template <int FMT, int WMODE>
__device__ __forceinline__ uint32_t stored_bits(const BuildFixed& b,
                                                const double* edge_w, bool exc,
                                                uint32_t tgt, uint32_t tie) {
  if (FMT == SNN_W_BF16_8B)
    return WMODE == 0 ? bf16_weight_bits(b, exc, tgt, tie)
                      : bf16_bits_rne(edge_w[tie]);
  return __float_as_uint(
      __double2float_rn(weight_of<WMODE>(b, edge_w, exc, tgt, tie)));
}

// Writes the row's synapses in the store's layout, its tile index and its
// part of the statistics.
template <int FMT, int WMODE>
__device__ void pack_row(const uint64_t* sorted, uint32_t len, uint32_t row,
                         uint64_t beg, const StoreOut& o, const BuildFixed& b,
                         const double* edge_w, TileGeom g, uint32_t n_tiles,
                         uint32_t* tile_off, uint32_t* stats,
                         const uint32_t* ends) {
  const bool exc = row < b.n_e;
  float wmax = 0.f;
  uint32_t run_max = 0, d_min = 0xFFFFFFFFu, d_max = 0;
  for (uint32_t p = threadIdx.x; p < len; p += blockDim.x) {
    uint64_t key = sorted[p];
    uint32_t d = key_delay(key, g);
    uint32_t tgt = key_target(key, g);
    uint32_t tie = (uint32_t)key;
    const uint32_t bits = stored_bits<FMT, WMODE>(b, edge_w, exc, tgt, tie);
    wmax = fmaxf(wmax, fabsf(FMT == SNN_W_BF16_8B ? bf16_to_f32(bits)
                                                  : __uint_as_float(bits)));
    d_min = min(d_min, d);
    d_max = max(d_max, d);
    const uint32_t in_tile = (uint32_t)(key >> 32) & ((1u << g.lb) - 1u);
    const uint32_t cell = (d - (uint32_t)o.d_base) * g.tw + in_tile;
    if (o.lay == kLayRecords) {
      if (FMT == SNN_W_FP32_12B) {
        uint32_t* r = reinterpret_cast<uint32_t*>(o.recs) + (beg + p) * 3u;
        r[0] = tgt;
        r[1] = bits;
        r[2] = d & 0xFFu;
      } else {
        reinterpret_cast<uint2*>(o.recs)[beg + p] =
            make_uint2(tgt, (d & 0xFFu) | (bits << 16));
      }
    } else if (FMT == SNN_W_FP32_12B) {
      o.wts[beg + p] = __uint_as_float(bits);
      o.tgts[beg + p] = tgt;
      o.cells[beg + p] = (uint16_t)cell;
    } else {
      uint32_t* r = reinterpret_cast<uint32_t*>(o.recs) + 2u * beg;
      r[len + p] = tgt;
      if (o.lay == kLayHom) {
        reinterpret_cast<uint16_t*>(r)[p] = (uint16_t)cell;
        reinterpret_cast<uint16_t*>(r)[len + p] = (uint16_t)bits;
      } else {
        r[p] = (cell & 0xFFFFu) |
               (o.lay == kLayI16 ? i16_bits(bf16_to_f32(bits), o.qs) : bits) << 16;
      }
    }
    // multiplicity of (target, delay): length of the run of equal keys
    // (ignoring the tie field) that starts here
    if (p == 0 || (sorted[p - 1] >> 32) != (key >> 32)) {
      uint32_t r = 1;
      while (p + r < len && (sorted[p + r] >> 32) == (key >> 32)) ++r;
      run_max = max(run_max, r);
    }
  }
  // |w| >= 0 orders like its bit pattern as an unsigned integer
  const uint32_t wbits = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(wmax));
  run_max = __reduce_max_sync(0xFFFFFFFFu, run_max);
  d_min = __reduce_min_sync(0xFFFFFFFFu, d_min);
  d_max = __reduce_max_sync(0xFFFFFFFFu, d_max);
  if ((threadIdx.x & 31u) == 0) {
    // the four words settle after a few rows: only a value beyond the
    // current one goes to the atomic (millions of warps would otherwise
    // queue on one line)
    const volatile uint32_t* st = stats;
    if (run_max > st[0]) atomicMax(&stats[0], run_max);
    if (wbits > st[1]) atomicMax(&stats[1], wbits);
    if (d_min < st[2]) atomicMin(&stats[2], d_min);
    if (d_max > st[3]) atomicMax(&stats[3], d_max);
  }
  // tile index: first position whose tile is >= tau (where the bucket before
  // ends, if the row was sorted by buckets; else by bisection)
  uint32_t* out = tile_off + (uint64_t)row * (n_tiles + 1);
  if (ends) {
    for (uint32_t tau = threadIdx.x; tau <= n_tiles; tau += blockDim.x)
      out[tau] = tau ? ends[tau - 1] : 0u;
    return;
  }
  for (uint32_t tau = threadIdx.x; tau <= n_tiles; tau += blockDim.x) {
    if (tau == n_tiles) {  // every key's tile is below n_tiles
      out[tau] = len;
      continue;
    }
    const uint64_t probe = (uint64_t)tau << (40 + g.lb);
    uint32_t lo = 0, hi = len;
    while (lo < hi) {
      uint32_t mid = (lo + hi) >> 1;
      if (sorted[mid] < probe) lo = mid + 1; else hi = mid;
    }
    out[tau] = lo;
  }
}

// In-place ascending bitonic sort of P (a power of two) keys.
__device__ void bitonic(uint64_t* a, uint32_t P) {
  for (uint32_t k = 2; k <= P; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t i = threadIdx.x; i < P; i += blockDim.x) {
        uint32_t l = i ^ j;
        if (l > i) {
          uint64_t x = a[i], y = a[l];
          bool up = (i & k) == 0;
          if ((x > y) == up) {
            a[i] = y;
            a[l] = x;
          }
        }
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ uint32_t pow2_ceil(uint32_t x) {
  uint32_t p = 1;
  while (p < x) p <<= 1;
  return p;
}

// Segments (keys of one target tile) up to this long are rank-sorted by a
// warp in registers; a row with a longer one is sorted whole (bitonic).
constexpr uint32_t kWarpSegMax = 256;
// Rows of stores with more tiles than this are sorted whole.
constexpr uint32_t kBucketTilesMax = 4096;

// Rank sort of one segment of up to 32 Q keys by a warp: a key's rank is the
// number of smaller keys (keys are distinct).
template <int Q>
__device__ __forceinline__ void rank_segment(uint64_t* a, uint32_t c) {
  const uint32_t lane = threadIdx.x & 31u;
  uint64_t key[Q];
  uint32_t rank[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    rank[q] = 0;
    key[q] = lane + 32u * q < c ? a[lane + 32u * q] : ~0ull;
  }
#pragma unroll 4
  for (uint32_t i = 0; i < c; ++i) {
    const uint64_t y = a[i];  // the same word for every lane
#pragma unroll
    for (int q = 0; q < Q; ++q) rank[q] += y < key[q];
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (lane + 32u * q < c) a[rank[q]] = key[q];
  __syncwarp();
}

// Sort one row of keys in shared memory (len keys at a[0..len), room for the
// next power of two; cnt: n_tiles + 1 words): bucket by target tile
// (histogram, exclusive scan by one warp, scatter from registers), then every
// warp rank-sorts the short segments of the tiles it takes, with as many
// registers a lane as the segment needs.  The result equals a full sort of
// the row; returns the buckets' ends.  Falls back to the bitonic network
// (returning null) when a segment is longer than kWarpSegMax or the store has
// too many tiles.
// The scan by one thread and eight compares a key for every segment, in CTAs
// of 1,024 threads of which one fits an SM, took 33 us a row of 3,000 keys.
__device__ const uint32_t* sort_row(uint64_t* a, uint32_t len, uint32_t* cnt,
                                    uint32_t n_tiles, int lb) {
  const uint32_t P = pow2_ceil(len);
  bool whole = n_tiles > kBucketTilesMax || len > 16u * blockDim.x;
  if (!whole) {
    __shared__ uint32_t s_max;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t n_warps = blockDim.x >> 5;
    for (uint32_t t = threadIdx.x; t <= n_tiles; t += blockDim.x) cnt[t] = 0;
    __syncthreads();
    // keys of this thread (at most 16) into registers, tiles counted
    uint64_t r[16];
#pragma unroll
    for (uint32_t q = 0; q < 16; ++q) {
      const uint32_t i = threadIdx.x + q * blockDim.x;
      if (i < len) {
        r[q] = a[i];
        atomicAdd(&cnt[(uint32_t)(r[q] >> (40 + lb))], 1u);
      }
    }
    __syncthreads();
    // longest segment, and the exclusive scan of the counts
    if (warp == 0) {
      uint32_t run = 0, mx = 0;
      for (uint32_t t0 = 0; t0 <= n_tiles; t0 += 32) {
        const uint32_t t = t0 + lane;
        const uint32_t c = t <= n_tiles ? cnt[t] : 0u;
        uint32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
          if (lane >= (uint32_t)o) inc += y;
        }
        if (t <= n_tiles) cnt[t] = run + inc - c;
        run += __shfl_sync(0xFFFFFFFFu, inc, 31);
        mx = max(mx, c);
      }
      mx = __reduce_max_sync(0xFFFFFFFFu, mx);
      if (lane == 0) s_max = mx;
    }
    __syncthreads();
    const uint32_t longest = s_max;
    whole = longest > kWarpSegMax;
    // scatter into the buckets (cnt becomes each bucket's end)
#pragma unroll
    for (uint32_t q = 0; q < 16; ++q) {
      const uint32_t i = threadIdx.x + q * blockDim.x;
      if (i < len) {
        const uint32_t pos = atomicAdd(&cnt[(uint32_t)(r[q] >> (40 + lb))], 1u);
        a[pos] = r[q];
      }
    }
    __syncthreads();
    if (!whole) {
      for (uint32_t t = warp; t < n_tiles; t += n_warps) {
        const uint32_t end = cnt[t];
        const uint32_t beg = t == 0 ? 0u : cnt[t - 1];
        const uint32_t c = end - beg;
        if (c < 2) continue;
        if (c <= 32) rank_segment<1>(a + beg, c);
        else if (c <= 64) rank_segment<2>(a + beg, c);
        else if (c <= 96) rank_segment<3>(a + beg, c);
        else if (c <= 128) rank_segment<4>(a + beg, c);
        else rank_segment<kWarpSegMax / 32>(a + beg, c);
      }
      __syncthreads();
      return cnt;
    }
  }
  for (uint32_t i = len + threadIdx.x; i < P; i += blockDim.x) a[i] = ~0ull;
  __syncthreads();
  if (P > 1) bitonic(a, P);
  return nullptr;
}

template <int FMT, int WMODE>
__global__ void __launch_bounds__(1024) k_sort_pack(uint32_t n, const uint64_t* row_ptr,
                            uint64_t* keys, StoreOut recs, BuildFixed b,
                            const double* edge_w, uint32_t cap, TileGeom g,
                            uint32_t n_tiles, uint32_t* tile_off,
                            uint32_t* stats) {
  extern __shared__ uint64_t sk[];
  uint32_t* cnt = reinterpret_cast<uint32_t*>(sk + cap);
  for (uint32_t row = blockIdx.x; row < n; row += gridDim.x) {
    const uint64_t beg = row_ptr[row];
    const uint32_t len = (uint32_t)(row_ptr[row + 1] - beg);
    if (len > cap) continue;                 // uniform per block
    for (uint32_t i = threadIdx.x; i < len; i += blockDim.x) sk[i] = keys[beg + i];
    __syncthreads();
    const uint32_t* ends = len > 1 ? sort_row(sk, len, cnt, n_tiles, g.lb) : nullptr;
    pack_row<FMT, WMODE>(sk, len, row, beg, recs, b, edge_w, g, n_tiles,
                         tile_off, stats, ends);
    __syncthreads();
  }
}

template <int FMT, int WMODE>
__global__ void __launch_bounds__(1024) k_sort_long(const uint32_t* rows, uint32_t n_long,
                            const uint64_t* row_ptr,
                            uint64_t* keys, StoreOut recs, BuildFixed b,
                            const double* edge_w, uint64_t* scratch,
                            const uint64_t* scratch_off, TileGeom g,
                            uint32_t n_tiles, uint32_t* tile_off,
                            uint32_t* stats) {
  for (uint32_t j = blockIdx.x; j < n_long; j += gridDim.x) {
    const uint32_t row = rows[j];
    const uint64_t beg = row_ptr[row];
    const uint32_t len = (uint32_t)(row_ptr[row + 1] - beg);
    uint64_t* a = scratch + scratch_off[j];
    const uint32_t P = pow2_ceil(len);
    for (uint32_t i = threadIdx.x; i < P; i += blockDim.x)
      a[i] = i < len ? keys[beg + i] : ~0ull;
    __syncthreads();
    bitonic(a, P);
    pack_row<FMT, WMODE>(a, len, row, beg, recs, b, edge_w, g, n_tiles,
                         tile_off, stats, nullptr);
    __syncthreads();
  }
}

template <int FMT>
__global__ void k_unpack(const void* recs, uint64_t n, uint32_t* tgt,
                         uint8_t* delay, float* w) {
  for (uint64_t s = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; s < n;
       s += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t t, d;
    float x;
    if (FMT == SNN_W_FP32_12B) {
      const uint32_t* p = reinterpret_cast<const uint32_t*>(recs) + s * 3u;
      t = p[0];
      x = __uint_as_float(p[1]);
      d = p[2] & 0xFFu;
    } else {
      uint2 r = reinterpret_cast<const uint2*>(recs)[s];
      t = r.x;
      d = r.y & 0xFFu;
      x = bf16_to_f32(r.y >> 16);
    }
    if (tgt) tgt[s] = t;
    if (delay) delay[s] = (uint8_t)d;
    if (w) w[s] = x;
  }
}

// The same for a split store, row by row: targets, and delays from the cells.
// What bounds it: memory; four synapses of a thread are read before any is
// written, and a warp writes whole lines of the outputs.  On whole records, one at a
// time from the row's start with a division each, and here: 1.27e9 synapses FP32
// 4,199, 4,406, 3,657 us (6.6 TB/s); 2.5e8 BF16 756, 828, 627 us.
__global__ void __launch_bounds__(256) k_unpack_split(NetView v, uint32_t* tgt,
                                                      uint8_t* delay, float* w) {
  constexpr uint32_t U = 4;
  const bool f32 = v.fmt == SNN_W_FP32_12B, hom = v.lay == kLayHom;
  const uint32_t magic = cell_magic(v.tile_w);
  for (uint32_t row = blockIdx.x; row < v.n_src; row += gridDim.x) {
    const uint64_t beg = v.row_ptr[row];
    const uint32_t len = (uint32_t)(v.row_ptr[row + 1] - beg);
    const uint32_t* r = reinterpret_cast<const uint32_t*>(v.recs) + 2u * beg;
    const uint16_t* r16 = reinterpret_cast<const uint16_t*>(r);
    const uint32_t off = (uint32_t)beg & 31u;
    for (uint32_t q0 = threadIdx.x; q0 < len + off; q0 += U * blockDim.x) {
      uint32_t cell[U], t[U], wb[U];
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) {
        const uint32_t p = q0 + u * blockDim.x - off;  // (before the row: >= len)
        if (p >= len) continue;
        if (f32) {
          if (delay) cell[u] = v.cells[beg + p];
          if (tgt) t[u] = v.tgts[beg + p];
          if (w) wb[u] = reinterpret_cast<const uint32_t*>(v.recs)[beg + p];
        } else {
          if (tgt) t[u] = r[len + p];
          cell[u] = hom ? r16[p] : r[p];
          if (hom && w) wb[u] = r16[len + p];
        }
      }
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) {
        const uint32_t p = q0 + u * blockDim.x - off;
        if (p >= len) continue;
        if (tgt) tgt[beg + p] = t[u];
        if (delay)
          delay[beg + p] =
              (uint8_t)(cell_step(cell[u] & 0xFFFFu, magic) + (uint32_t)v.d_base);
        if (w)
          w[beg + p] = f32 ? __uint_as_float(wb[u])
                       : hom ? __uint_as_float(wb[u] << 16)
                       : v.lay == kLayI16 ? i16_weight(cell[u], v.acc_qs_min)
                                          : __uint_as_float(cell[u] & 0xFFFF0000u);
      }
    }
  }
}

unsigned grid_for(uint64_t n, unsigned threads) {
  uint64_t b = (n + threads - 1) / threads;
  if (b > 65536u * 8u) b = 65536u * 8u;
  return b ? (unsigned)b : 1u;
}

// Build mode of the calling thread, set around a build by the API
// (snn_params.build_yield).
thread_local unsigned t_build_yield = 0;

// Launch shape of a build kernel.  Normal: the kernel's own grid.
// Yielding: the same grid of short CTAs (one target or one row each), but of
// 1024 threads and with more than half of an SM's shared memory, so that no
// two share an SM.  Each SM then becomes entirely free whenever one of its
// build CTAs ends (every few to a few hundred microseconds), and the CTA
// scheduler hands it to pending work of higher-priority streams first: the
// kernels of running nets, whose delivery CTAs need a whole SM and would
// otherwise wait for the build to end, since small build CTAs keep refilling
// partly free SMs.
struct BuildShape {
  unsigned blocks, threads;
  size_t smem;
};

template <class Kernel>
cudaError_t build_shape(Kernel kernel, unsigned blocks, unsigned threads,
                        size_t smem, BuildShape* out) {
  *out = BuildShape{blocks, threads, smem};
  int dev = 0, per_sm = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  // the kernel's dynamic shared-memory limit is always raised to all that
  // its static shared memory leaves of the opt-in amount: one value for
  // every caller, so that builds on several host threads never lower it
  // under one another's launch
  cudaFuncAttributes fa;
  if ((e = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return e;
  const int dyn_max = optin - (int)fa.sharedSizeBytes;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           dyn_max);
  if (e != cudaSuccess) return e;
  if (!t_build_yield) return cudaSuccess;
  const size_t excl = std::min<size_t>((size_t)per_sm / 2 + 2048, (size_t)dyn_max);
  out->threads = threads > 1024 ? threads : 1024;
  out->smem = std::max(smem, excl);
  return cudaSuccess;
}

template <int FMT, int WMODE>
cudaError_t sort_pack_t(uint32_t n, const uint64_t* row_ptr, uint64_t* keys,
                        StoreOut recs, const BuildFixed* b, const double* edge_w,
                        uint32_t max_row, const uint32_t* long_rows,
                        uint32_t n_long, uint64_t* long_scratch,
                        const uint64_t* long_off, TileGeom g, uint32_t n_tiles,
                        uint32_t* tile_off, uint32_t* stats, cudaStream_t s) {
  BuildFixed bb = b ? *b : BuildFixed{};
  uint32_t cap = max_row < kSortCap ? max_row : kSortCap;
  uint32_t P = 1;
  while (P < cap) P <<= 1;
  // keys (room for the next power of two) and the tile buckets
  size_t smem = (size_t)P * sizeof(uint64_t) +
                (size_t)(std::min(n_tiles, kBucketTilesMax) + 1) * sizeof(uint32_t);
  cudaError_t e;
  // 16 keys a thread at most: a CTA waits for itself several times a row, so
  // several small ones on an SM keep it busy
  unsigned threads = std::max(128u, std::min(1024u, P / 16u));
  unsigned blocks = n < (1u << 20) ? n : (1u << 20);
  BuildShape sh;
  if (blocks) {
    if ((e = build_shape(k_sort_pack<FMT, WMODE>, blocks, threads, smem, &sh)) !=
        cudaSuccess)
      return e;
    k_sort_pack<FMT, WMODE><<<sh.blocks, sh.threads, sh.smem, s>>>(
        n, row_ptr, keys, recs, bb, edge_w, P, g, n_tiles, tile_off, stats);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (n_long) {
    if ((e = build_shape(k_sort_long<FMT, WMODE>, n_long, 1024, 0, &sh)) !=
        cudaSuccess)
      return e;
    k_sort_long<FMT, WMODE><<<sh.blocks, sh.threads, sh.smem, s>>>(
        long_rows, n_long, row_ptr, keys, recs, bb, edge_w, long_scratch,
        long_off, g, n_tiles, tile_off, stats);
  }
  return cudaGetLastError();
}

}  // namespace

void set_build_yield(unsigned on) { t_build_yield = on; }

// Whether the fixed rule's count runs in shared memory (*bytes of it a CTA,
// *parts CTAs): not in a build that yields SMs, for populations past shared
// memory, for counts that could pass 16 bits, or for too few synapses to pay
// for clearing and adding up the counters.
static cudaError_t count_shared(const BuildFixed& b, uint32_t n_src, bool* use,
                                bool* w16, size_t* bytes, uint32_t* parts) {
  *use = false;
  const uint64_t syn = (uint64_t)b.n_tgt * (b.k_e + b.k_i);
  if (t_build_yield || syn < (4ull << 20) || syn < 64ull * n_src) return cudaSuccess;
  int dev = 0, sms = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  *w16 = (size_t)n_src * 4 > (size_t)optin;
  *bytes = *w16 ? ((size_t)n_src + 1) / 2 * 4 : (size_t)n_src * 4;
  *parts = std::min<uint32_t>((uint32_t)std::max(sms, 1), b.n_tgt);
  // a source's draws in a CTA are binomial: a mean of 2^14 leaves 2^16 out of
  // reach
  const double per = std::ceil((double)b.n_tgt / *parts);
  *use = *bytes <= (size_t)optin &&
         (!b.n_e || per * b.k_e / b.n_e <= 16384.0) &&
         (!b.n_i || per * b.k_i / b.n_i <= 16384.0);
  return cudaSuccess;
}

cudaError_t build_count_fixed(const BuildFixed& b, uint32_t n_src, uint32_t* deg,
                              cudaStream_t s) {
  if (b.n_tgt == 0 || b.k_e + b.k_i == 0) return cudaSuccess;
  bool use = false, w16 = false;
  size_t bytes = 0;
  uint32_t parts = 0;
  cudaError_t e = count_shared(b, n_src, &use, &w16, &bytes, &parts);
  if (e != cudaSuccess) return e;
  BuildShape sh;
  if (use) {
    const uint32_t per = (b.n_tgt + parts - 1) / parts;
    // (build_shape raises the kernel's shared-memory limit)
    e = w16 ? build_shape(k_count_shared<true>, parts, 1024, bytes, &sh)
            : build_shape(k_count_shared<false>, parts, 1024, bytes, &sh);
    if (e != cudaSuccess) return e;
    if (w16)
      k_count_shared<true><<<sh.blocks, sh.threads, sh.smem, s>>>(b, n_src, per, deg);
    else
      k_count_shared<false><<<sh.blocks, sh.threads, sh.smem, s>>>(b, n_src, per, deg);
    return cudaGetLastError();
  }
  e = build_shape(k_count_fixed, b.n_tgt, 256, 0, &sh);
  if (e != cudaSuccess) return e;
  k_count_fixed<<<sh.blocks, sh.threads, sh.smem, s>>>(b, deg);
  return cudaGetLastError();
}

cudaError_t build_scatter_fixed(const BuildFixed& b, const uint64_t* row_ptr,
                                uint32_t* cursor, uint64_t* keys,
                                uint32_t tile_w, int lo_bits, cudaStream_t s) {
  if (b.n_tgt == 0 || b.k_e + b.k_i == 0) return cudaSuccess;
  BuildShape sh;
  cudaError_t e = build_shape(k_scatter_fixed, b.n_tgt, 256, 0, &sh);
  if (e != cudaSuccess) return e;
  k_scatter_fixed<<<sh.blocks, sh.threads, sh.smem, s>>>(
      b, row_ptr, cursor, keys, TileGeom{tile_w, lo_bits});
  return cudaGetLastError();
}

cudaError_t build_count_edges(const uint32_t* src, uint64_t n, uint32_t* deg,
                              cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_count_edges<<<grid_for(n, 256), 256, 0, s>>>(src, n, deg);
  return cudaGetLastError();
}

cudaError_t build_scatter_edges(const uint32_t* src, const uint32_t* tgt,
                                const uint8_t* delay, uint64_t n,
                                const uint64_t* row_ptr, uint32_t* cursor,
                                uint64_t* keys, uint32_t tile_w, int lo_bits,
                                cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_scatter_edges<<<grid_for(n, 256), 256, 0, s>>>(
      src, tgt, delay, n, row_ptr, cursor, keys, TileGeom{tile_w, lo_bits});
  return cudaGetLastError();
}

cudaError_t build_sort_pack(int fmt, uint32_t n, const uint64_t* row_ptr,
                            uint64_t* keys, StoreOut recs, const BuildFixed* b,
                            const double* edge_w, uint32_t max_row,
                            const uint32_t* long_rows, uint32_t n_long,
                            uint64_t* long_scratch,
                            const uint64_t* long_scratch_off, uint32_t tile_w,
                            int lo_bits, uint32_t n_tiles, uint32_t* tile_off,
                            uint32_t* stats, cudaStream_t s) {
  const TileGeom g{tile_w, lo_bits};
#define SNN_SORT_ARGS                                                       \
  n, row_ptr, keys, recs, b, edge_w, max_row, long_rows, n_long,           \
      long_scratch, long_scratch_off, g, n_tiles, tile_off, stats, s
  if (fmt == SNN_W_FP32_12B)
    return edge_w ? sort_pack_t<SNN_W_FP32_12B, 1>(SNN_SORT_ARGS)
                  : sort_pack_t<SNN_W_FP32_12B, 0>(SNN_SORT_ARGS);
  return edge_w ? sort_pack_t<SNN_W_BF16_8B, 1>(SNN_SORT_ARGS)
                : sort_pack_t<SNN_W_BF16_8B, 0>(SNN_SORT_ARGS);
#undef SNN_SORT_ARGS
}

cudaError_t unpack_store(const NetView& v, uint64_t n_syn, uint32_t* tgt,
                         uint8_t* delay, float* w, cudaStream_t s) {
  if (n_syn == 0) return cudaSuccess;
  if (v.lay != kLayRecords)
    k_unpack_split<<<std::min(v.n_src, 1u << 16), 256, 0, s>>>(v, tgt, delay, w);
  else if (v.fmt == SNN_W_FP32_12B)
    k_unpack<SNN_W_FP32_12B><<<grid_for(n_syn, 256), 256, 0, s>>>(
        v.recs, n_syn, tgt, delay, w);
  else
    k_unpack<SNN_W_BF16_8B><<<grid_for(n_syn, 256), 256, 0, s>>>(
        v.recs, n_syn, tgt, delay, w);
  return cudaGetLastError();
}

}  // namespace snn
