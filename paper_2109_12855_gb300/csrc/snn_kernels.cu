// snn_kernels.cu -- the simulation hot path on sm_103a.
//
//  k_update   fused neuron update for one min-delay interval (Section 2.1 of
//             arXiv 2109.12855: exact integration of the linear
//             subthreshold dynamics on the 0.1 ms grid), ring-buffer slot
//             read-and-clear, Poisson drive, threshold/reset/refractoriness,
//             and warp-ballot compaction of the spikes into the interval
//             list.  Each compacted spike also reserves its source row's
//             chunks with the same 64-bit atomic, so the list carries an
//             exclusive prefix sum of chunk counts in list order (the
//             degree scan of the load-balanced expansion) with no extra pass.
//  k_deliver  spike delivery (Section 3.2, Algorithm REF): every spike's
//             target segment is expanded and each synapse adds its weight
//             into rb[(t + delay) mod S][target].  Load balance is a
//             merge-path split of the interval's chunk space: warp w takes
//             chunks [w C / W, (w+1) C / W), finds its first spike by a
//             32-ary search of the prefix sums, then walks spikes and
//             chunks.  Each lane reads its records with 16-byte loads
//             (streaming cache hint); additions are red.global.add.f32.
//  k_deliver_tiled  the default delivery (Section 3.2's target-ordered
//             access, made tile-local): one CTA per tile of targets sums
//             the interval's events for its targets in shared memory in
//             exact fixed point, then adds them into its window of the ring
//             buffer, one reduction a cell.
//  k_simulate  update, exchange and delivery of many intervals in one
//             cooperative launch, for nets of at most a tile per SM.
//  k_update_batch, k_deliver_tiled_batch  the same for all nets of a served
//             batch in one launch each.
//  k_prepare_external  prefix sum of chunk counts for a caller's list.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>

#include "snn_internal.cuh"

namespace snn {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kUpdThreads = 256;
constexpr int kDelThreads = 256;

__device__ __forceinline__ void red_add_f32(float* p, float v) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

__device__ __forceinline__ uint4 ld_stream16(const void* p) {
  return __ldcs(reinterpret_cast<const uint4*>(p));
}

// ---------------------------------------------------------------------------
// Initial state.
// ---------------------------------------------------------------------------
__global__ void k_init_state(NetView v, float v_reset, float v_span,
                            uint64_t seed, int random) {
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= v.n) return;
  float V0 = 0.0f;
  if (random) {
    U4 r = draw(seed, v.g0 + i, 0, 1u);  // keyed by the global index
    double u = (double)r.x * 0x1p-32;
    V0 = (float)((double)v_reset + (double)v_span * u);
  }
  v.V[i] = V0;
  v.I[i] = 0.0f;
  v.J[i] = 0.0f;
  v.refr[i] = 0;
}

__global__ void k_list_to_arrays(const SpikeEntry* list, uint64_t n,
                                 uint32_t* src, int32_t* t) {
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < n;
       k += (uint64_t)gridDim.x * blockDim.x) {
    src[k] = list[k].src;
    t[k] = list[k].t;
  }
}

__global__ void k_fill_i32(int32_t* p, int32_t value, uint64_t n) {
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < n;
       k += (uint64_t)gridDim.x * blockDim.x)
    p[k] = value;
}

// ---------------------------------------------------------------------------
// Fused update.
//
// One thread per neuron integrates its state for the interval's steps, in the
// 4-step blocks that the drive is drawn in: a block's ring-buffer loads, draws
// and table look-ups are independent and issued together, then its steps run in
// order.  What bounds it: issue, where several waves of blocks hide the
// latencies (562,500 neurons, 10 steps: 1,240 warp instructions a warp without
// spikes, 1,440 with an interval's spikes, 66 % of the issue slots), else the latency of a
// thread's chain.
// Spikes are kept as a per-thread bit mask of step indices and compacted once
// per warp for up to 32 steps: a warp scan of the per-thread counts, then one
// set of global atomics per warp with spikes reserves its list entries and
// chunk ranges.
// ---------------------------------------------------------------------------

// Plasticity state at a spike of excitatory neuron i at step t: the
// presynaptic trace (kept with the values before this spike, which its own
// delivery needs) and the postsynaptic ring of the last hist spikes with the
// trace right after each.  Traces decay by exp(-steps h / tau) and jump by 1.
__device__ __forceinline__ void stdp_on_spike(const StdpView& sp, uint32_t i,
                                              int32_t t, uint32_t pitch) {
  const int32_t tl = sp.pre_t[i];
  const float kl = sp.pre_k[i];
  sp.prev_t[i] = tl;
  sp.prev_k[i] = kl;
  sp.pre_k[i] =
      (tl == kNoSpike ? 0.f : kl * exp2f(-(float)(t - tl) * sp.l2_plus)) + 1.f;
  sp.pre_t[i] = t;
  const uint32_t n = sp.ring_n[i];
  const uint32_t hm = sp.hist - 1u;
  float km = 0.f;
  if (n) {
    const size_t last = (size_t)((n - 1u) & hm) * pitch + i;
    km = sp.ring_k[last] * exp2f(-(float)(t - sp.ring_t[last]) * sp.l2_minus);
  }
  const size_t slot = (size_t)(n & hm) * pitch + i;
  sp.ring_t[slot] = t;
  sp.ring_k[slot] = km + 1.f;
  sp.ring_n[i] = n + 1u;
}

// L2 prefetch of source src's row of the tile index, line by line.
__device__ __forceinline__ void prefetch_row_l2(const NetView& v, uint32_t src) {
  const char* a = reinterpret_cast<const char*>(
      v.tile_off + (uint64_t)src * (v.n_tiles + 1u));
  const char* e = a + 4ull * (v.n_tiles + 1u);
  for (const char* p = reinterpret_cast<const char*>(
           reinterpret_cast<uintptr_t>(a) & ~(uintptr_t)127);
       p < e; p += 128)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// One step of a neuron: exact integration, this step's input (ring buffer and
// drive), threshold.  Returns whether it fired.
__device__ __forceinline__ bool update_step(const UpdConst& c, float& V, float& I,
                                            float& J, int& refr, float in) {
  // (1) membrane, unless refractory
  if (refr == 0) V = c.p31 * J + c.p32 * I + c.p33 * V;
  else refr -= 1;
  // (2) synaptic current and its derivative
  I = c.p21 * J + c.p22 * I;
  J = c.p11 * J;
  // (3) input
  J += c.psc * in;
  // (4) threshold
  if (!(V >= c.v_th)) return false;
  V = c.v_reset;
  refr = c.refr_steps;
  return true;
}

// Body of the update for neuron block `block` of net v (one thread per
// neuron); shared by the single-net and the batched kernels.
// PL: the single-net update, which also keeps the plasticity state and the
// long-run spike statistics (the batched serving update does neither).
// ONE: the grid is one wave, whose latency counts: the neurons' spike
// statistics are read before the integration, so that those that fire need not
// wait for them.
template <bool PL, bool ONE>
__device__ __forceinline__ void update_body(const NetView& v, const UpdConst& c,
                                            int n_steps, int from_ctl,
                                            long long t0_arg, uint32_t block) {
  __shared__ uint32_t s_thr[kMaxPoisson];
  __shared__ uint8_t s_guide[256];
  for (int k = threadIdx.x; k < c.n_thr; k += blockDim.x) s_thr[k] = c.thr[k];
  for (int k = threadIdx.x; k < 256; k += blockDim.x) s_guide[k] = c.guide[k];

  const uint32_t i = block * blockDim.x + threadIdx.x;
  const bool live = i < v.n;
  float V = 0.f, I = 0.f, J = 0.f;
  int refr = 0;
  uint32_t nch = 0;
  unsigned long long deg = 0;
  if (live) {
    V = v.V[i];
    I = v.I[i];
    J = v.J[i];
    refr = v.refr[i];
    // the neuron's own row (rows are indexed by global source)
    uint64_t beg = v.row_ptr[v.g0 + i], end = v.row_ptr[v.g0 + i + 1];
    nch = row_chunks(beg, end, v.chunk);
    deg = end - beg;
  }
  int32_t isi_last = kNoSpike;
  uint32_t isi_spk = 0, isi_cnt = 0;
  double isi_s1 = 0.0, isi_s2 = 0.0;
  auto load_isi = [&]() {
    isi_last = v.isi_last[i];
    isi_spk = v.isi_spikes[i];
    isi_cnt = v.isi_n[i];
    isi_s1 = v.isi_sum[i];
    isi_s2 = v.isi_sq[i];
  };
  if (PL && ONE && live && v.isi_spikes) load_isi();
  // the single-net update may start while the previous kernel's last CTAs
  // run (programmatic dependent launch): everything above reads only what no
  // kernel that can directly precede it writes -- a delivery adds to the ring
  // buffer, and a launch of k_simulate, which writes state and statistics, is
  // followed by a fully ordered memset (launch_simulate_t); from here on the
  // delivery's ring-buffer additions, clock and counters must be complete
  if constexpr (PL) asm volatile("griddepcontrol.wait;" ::: "memory");
  const long long t0 = from_ctl ? v.ctl->t_now : t0_arg;
  if (block == 0 && threadIdx.x == 0) {
    v.ctl->iv_steps = n_steps;
    if (!from_ctl) v.ctl->t_now = t0;
  }
  __syncthreads();
  float* const rb_i = v.rb + i;  // slot s of neuron i at rb_i[s * pitch]

  for (int s0 = 0; s0 < n_steps; s0 += 32) {
    const int ns = n_steps - s0 < 32 ? n_steps - s0 : 32;
    uint32_t mask = 0;
    {
      const long long tc = t0 + s0;
      for (long long b = tc >> 2; 4 * b < tc + ns; ++b) {
        const int s1 = (int)(4 * b - tc);  // the block's first step, from tc
        float in[4];
        uint32_t k[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          in[q] = 0.f;
          if (live && s1 + q >= 0 && s1 + q < ns)
            in[q] = rb_i[((uint32_t)(tc + s1 + q) & v.slot_mask) * v.pitch];
        }
        if (c.n_thr > 0) {
          const U4 r = draw(c.seed, v.g0 + i, (uint64_t)b, 2u);  // by global index
          const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) k[q] = s_guide[w[q] >> 24];
          uint32_t th[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) th[q] = s_thr[k[q]];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if ((int)k[q] < c.n_thr - 1 && w[q] >= th[q]) {
              ++k[q];
              while ((int)k[q] < c.n_thr - 1 && w[q] >= s_thr[k[q]]) ++k[q];
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int st = s1 + q;
          if (!live || st < 0 || st >= ns) continue;
          if (c.n_thr > 0) in[q] += c.w_ext * (float)(int)k[q];
          rb_i[((uint32_t)(tc + st) & v.slot_mask) * v.pitch] = 0.0f;
          if (update_step(c, V, I, J, refr, in[q])) mask |= 1u << st;
        }
      }
    }
    // warp compaction of this chunk's spikes: a warp with spikes scans its
    // lanes' counts and reserves its list entries, chunk ranges and log
    // slots with one set of global atomics; warps without spikes (most of
    // them at a few Hz) go on without waiting for anyone
    const uint32_t cnt = __popc(mask);
    if (__ballot_sync(kFull, cnt != 0)) {
      const unsigned lane = threadIdx.x & 31u;
      // (several waves: only the statistics of the neurons that fired, whose
      // latency then overlaps the reservation; 24 bytes a neuron and interval
      // less)
      const bool isi = PL && cnt && v.isi_spikes;
      if (isi && !ONE) load_isi();
      uint32_t inc_cnt = cnt, inc_ch = cnt * nch;
      unsigned long long inc_deg = (unsigned long long)cnt * deg;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t ya = __shfl_up_sync(kFull, inc_cnt, o);
        const uint32_t yb = __shfl_up_sync(kFull, inc_ch, o);
        const unsigned long long yc = __shfl_up_sync(kFull, inc_deg, o);
        if (lane >= (unsigned)o) {
          inc_cnt += ya;
          inc_ch += yb;
          inc_deg += yc;
        }
      }
      const uint32_t ex_cnt = inc_cnt - cnt, ex_ch = inc_ch - cnt * nch;
      unsigned long long old = 0ull, logb = 0ull;
      uint32_t xbase = 0u;
      if (lane == 31u) {  // the warp's totals
        // all counters first (separate lines, the returning atomics in
        // flight together), then the overflow check on the list's one
        old = atomicAdd(&v.ctl->pair, ((unsigned long long)inc_cnt << 32) | inc_ch);
        logb = v.log_cap ? atomicAdd(&v.ctl->log_count, (unsigned long long)inc_cnt)
                         : 0ull;
        xbase = v.xbuf ? atomicAdd(v.xbuf, inc_cnt) : 0u;
        atomicAdd(&v.ctl->pending_events, inc_deg);
        atomicAdd(&v.ctl->spikes, (unsigned long long)inc_cnt);
        if ((uint32_t)old + (unsigned long long)inc_ch > 0xFFFFFFFFull)
          atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_CHUNKS);
      }
      old = __shfl_sync(kFull, old, 31);
      logb = __shfl_sync(kFull, logb, 31);
      xbase = __shfl_sync(kFull, xbase, 31);
      uint32_t m = mask, k = 0;
      while (m) {
        const int b = __ffs(m) - 1;
        m &= m - 1u;
        const long long t = t0 + s0 + b;
        const unsigned long long idx = (old >> 32) + ex_cnt + k;
        if (idx < v.list_cap) {
          SpikeEntry e;
          e.src = v.g0 + i;
          e.t = (int32_t)t;
          e.choff = (uint32_t)old + ex_ch + k * nch;
          e.pad = 0;
          v.list[idx] = e;
          // the tiled delivery that follows reads this source's row of the
          // tile index (two words per CTA): bring the row into L2 now
          if (v.tile_off && k == 0) prefetch_row_l2(v, v.g0 + i);
        } else {
          atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_SPIKE_LIST);
        }
        if (v.xbuf) {  // the partition exchange's copy of the list
          const uint32_t xi = xbase + ex_cnt + k;
          if (xi < v.xcap) {
            reinterpret_cast<uint2*>(v.xbuf + 4)[xi] =
                make_uint2(v.g0 + i, (uint32_t)(int32_t)t);
          } else {
            atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_SPIKE_LIST);
          }
        }
        if (v.log_cap) {
          const unsigned long long li = logb + ex_cnt + k;
          if (li < v.log_cap) {
            v.log_src[li] = v.g0 + i;
            v.log_t[li] = (int32_t)t;
          } else {
            atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_SPIKE_LOG);
          }
        }
        if (PL && v.plastic && i < v.sp.n_exc)
          stdp_on_spike(v.sp, i, (int32_t)t, v.pitch);
        if (isi) {
          if (isi_last != kNoSpike) {
            const double d = (double)((int32_t)t - isi_last);  // exact in FP64
            isi_s1 += d;
            isi_s2 += d * d;
            isi_cnt += 1u;
          }
          isi_last = (int32_t)t;
          isi_spk += 1u;
        }
        ++k;
      }
      if (isi) {
        v.isi_last[i] = isi_last;
        v.isi_spikes[i] = isi_spk;
        v.isi_n[i] = isi_cnt;
        v.isi_sum[i] = isi_s1;
        v.isi_sq[i] = isi_s2;
      }
    }
  }
  if (live) {
    v.V[i] = V;
    v.I[i] = I;
    v.J[i] = J;
    v.refr[i] = refr;
  }
}

// MINB blocks per SM: 3 leaves room for spill-free registers (a
// 112,500-neuron net's 440 blocks run in one wave); nets that need several
// waves anyway take 4, for more warps per SM.
template <int MINB>
__global__ void __launch_bounds__(kUpdThreads, MINB)
k_update(NetView v, UpdConst c, int n_steps, int from_ctl, long long t0_arg) {
  update_body<true, MINB == 3>(v, c, n_steps, from_ctl, t0_arg, blockIdx.x);
}

// Copies *src (of whole words) to shared memory, all threads of the CTA.
template <class T>
__device__ __forceinline__ void load_shared(T* dst, const T* src) {
  static_assert(sizeof(T) % 4 == 0, "whole words");
  for (uint32_t k = threadIdx.x; k < sizeof(T) / 4; k += blockDim.x)
    reinterpret_cast<uint32_t*>(dst)[k] = reinterpret_cast<const uint32_t*>(src)[k];
}

// All nets of a batch in one launch: block b updates neuron block bmap[b].y
// of net bmap[b].x, from that net's clock.
__global__ void __launch_bounds__(kUpdThreads, 3)
k_update_batch(const BatchNet* __restrict__ nets, const uint2* __restrict__ bmap) {
  __shared__ UpdConst s_c;
  __shared__ NetView s_v;
  const uint2 m = bmap[blockIdx.x];
  const BatchNet& bn = nets[m.x];
  load_shared(&s_c, &bn.c);
  load_shared(&s_v, &bn.v);
  const int n_steps = bn.n_steps;
  __syncthreads();
  update_body<false, true>(s_v, s_c, n_steps, 1, 0, m.y);  // served nets are static
}

// ---------------------------------------------------------------------------
// Delivery.
// ---------------------------------------------------------------------------
template <int FMT> struct Loaded;
template <> struct Loaded<SNN_W_FP32_12B> { uint4 a, b, c; };
template <> struct Loaded<SNN_W_BF16_8B> { uint4 a; };

template <int FMT>
__device__ __forceinline__ Loaded<FMT> load_lane(const void* recs,
                                                 uint64_t rec_index);
template <>
__device__ __forceinline__ Loaded<SNN_W_FP32_12B> load_lane<SNN_W_FP32_12B>(
    const void* recs, uint64_t r) {
  const char* p = reinterpret_cast<const char*>(recs) + r * 12u;
  Loaded<SNN_W_FP32_12B> x;
  x.a = ld_stream16(p);
  x.b = ld_stream16(p + 16);
  x.c = ld_stream16(p + 32);
  return x;
}
template <>
__device__ __forceinline__ Loaded<SNN_W_BF16_8B> load_lane<SNN_W_BF16_8B>(
    const void* recs, uint64_t r) {
  Loaded<SNN_W_BF16_8B> x;
  x.a = ld_stream16(reinterpret_cast<const char*>(recs) + r * 8u);
  return x;
}

// Record q (0 .. kPerLane-1) of a lane's loaded bytes.
template <int FMT>
__device__ __forceinline__ void unpack(const Loaded<FMT>& x, int q,
                                       uint32_t& tgt, uint32_t& d, float& w);
template <>
__device__ __forceinline__ void unpack<SNN_W_FP32_12B>(
    const Loaded<SNN_W_FP32_12B>& x, int q, uint32_t& tgt, uint32_t& d,
    float& w) {
  // 48 bytes = words a.x a.y a.z a.w b.x ... c.w; record q = words 3q..3q+2
  uint32_t wd[12] = {x.a.x, x.a.y, x.a.z, x.a.w, x.b.x, x.b.y,
                     x.b.z, x.b.w, x.c.x, x.c.y, x.c.z, x.c.w};
  tgt = wd[3 * q];
  w = __uint_as_float(wd[3 * q + 1]);
  d = wd[3 * q + 2] & 0xFFu;
}
template <>
__device__ __forceinline__ void unpack<SNN_W_BF16_8B>(
    const Loaded<SNN_W_BF16_8B>& x, int q, uint32_t& tgt, uint32_t& d,
    float& w) {
  uint32_t t0 = q == 0 ? x.a.x : x.a.z;
  uint32_t m0 = q == 0 ? x.a.y : x.a.w;
  tgt = t0;
  d = m0 & 0xFFu;
  w = __uint_as_float(m0 & 0xFFFF0000u);
}

// Bounds-checked builds: a record whose target lies outside [lo, lo + width)
// (or the net) or whose delay lies outside the store's range is skipped
// and flagged.  Production builds compile this to `true`.
__device__ __forceinline__ bool rec_in_bounds(const NetView& v, uint32_t tgt,
                                              uint32_t d, uint32_t lo,
                                              uint32_t width) {
  if (!kChecked) return true;
  const bool ok = tgt - lo < width && tgt < v.n && d >= (uint32_t)v.d_min &&
                  d <= (uint32_t)v.d_max;
  if (!ok) atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_CHECK);
  return ok;
}

template <int FMT, bool COUNT>
__global__ void __launch_bounds__(kDelThreads)
k_deliver(NetView v, unsigned long long* pair_p, unsigned int* done_p,
          const SpikeEntry* __restrict__ list, int advance_time) {
  constexpr int CH = Fmt<FMT>::kChunk;
  constexpr int PL = Fmt<FMT>::kPerLane;
  constexpr int G = FMT == SNN_W_FP32_12B ? 4 : 8;  // chunks in flight / warp
  __shared__ unsigned long long s_pair;
  if (threadIdx.x == 0) s_pair = *reinterpret_cast<volatile unsigned long long*>(pair_p);
  __syncthreads();
  const uint32_t n_sp = (uint32_t)(s_pair >> 32);
  const uint64_t n_ch = (uint32_t)s_pair;
  const unsigned lane = threadIdx.x & 31u;
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t c_begin = warp * n_ch / n_warps;
  const uint64_t c_end = (warp + 1) * n_ch / n_warps;

  if (c_begin < c_end) {
    // last spike j with choff[j] <= c_begin (choff is non-decreasing)
    uint32_t lo = 0, hi = n_sp;
    while (hi - lo > 32) {
      uint32_t p = lo + (uint32_t)(((uint64_t)(hi - lo) * lane) >> 5);
      bool le = list[p].choff <= c_begin;
      unsigned m = __ballot_sync(kFull, le);
      int last = 31 - __clz(m);
      uint32_t nlo = __shfl_sync(kFull, p, last);
      uint32_t nhi = __shfl_sync(kFull, p, last < 31 ? last + 1 : 31);
      lo = nlo;
      hi = last < 31 ? nhi : hi;
    }
    {
      uint32_t p = lo + lane;
      bool le = p < hi && list[p].choff <= c_begin;
      unsigned m = __ballot_sync(kFull, le);
      lo = lo + (31 - __clz(m));
    }
    uint32_t j = lo;
    uint64_t c = c_begin;
    uint32_t prev_choff = 0u;
    while (c < c_end && j < n_sp) {
      const SpikeEntry e = list[j];
      ++j;
      if (kChecked) {  // the merge-path split needs non-decreasing offsets
        if (e.choff < prev_choff) {
          atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_CHECK);
          break;
        }
        prev_choff = e.choff;
      }
      if (e.src >= v.n_src) continue;
      const uint64_t beg = v.row_ptr[e.src], end = v.row_ptr[e.src + 1];
      const uint64_t last = (uint64_t)e.choff + row_chunks(beg, end, CH);
      const uint64_t stop = last < c_end ? last : c_end;
      if (c < e.choff) c = e.choff;   // (only if entries were skipped)
      const int64_t abs0 = (int64_t)(beg / CH) - (int64_t)e.choff;
      const int32_t t = e.t;
      for (; c < stop; c += G) {
        Loaded<FMT> x[G];
#pragma unroll
        for (int g = 0; g < G; ++g)
          if (c + g < stop)
            x[g] = load_lane<FMT>(v.recs,
                                  (uint64_t)(abs0 + (int64_t)(c + g)) * CH +
                                      lane * PL);
#pragma unroll
        for (int g = 0; g < G; ++g) {
          if (c + g < stop) {
            const uint64_t r0 =
                (uint64_t)(abs0 + (int64_t)(c + g)) * CH + lane * PL;
#pragma unroll
            for (int q = 0; q < PL; ++q) {
              const uint64_t r = r0 + q;
              if (r >= beg && r < end) {
                uint32_t tgt, d;
                float w;
                unpack<FMT>(x[g], q, tgt, d, w);
                if (!rec_in_bounds(v, tgt, d, 0u, v.n)) continue;
                const size_t cell =
                    (size_t)(((uint32_t)t + d) & v.slot_mask) * v.pitch + tgt;
                red_add_f32(v.rb + cell, w);
                if (COUNT) atomicAdd(v.counts + cell, 1u);
              }
            }
          }
        }
      }
      c = stop;
    }
  }

  // The last CTA to finish clears the list counters for the next interval
  // (every CTA read them before arriving here) and advances the clock.
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    unsigned prev = atomicAdd(done_p, 1u);
    if (prev == gridDim.x - 1) {
      *pair_p = 0ull;
      *done_p = 0u;
      if (advance_time) {  // the interval's own list: commit its events
        if (v.xbuf) *v.xbuf = 0u;  // the next update refills the exchange list
        v.ctl->t_now += v.ctl->iv_steps;
        v.ctl->events += v.ctl->pending_events;
        v.ctl->pending_events = 0ull;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Tile-binned delivery.
//
// CTA tau owns the targets [tau TW, (tau+1) TW) and accumulates, in shared
// memory, every event of the list aimed at them for the ring steps
// base .. base + window - 1 that one interval can reach (base = interval
// start + min delay).  Rows are sorted by target tile, so the synapses of
// spike j for tile tau are one contiguous run, located by the row's tile
// index.  (A) the CTA describes a batch of runs in shared memory; (B) its 32
// warps take 32 / 2^lg runs at a time, 2^lg lanes a run; a lane reads aligned
// 16-byte vectors of its run (the store's split layouts, snn_internal.cuh: 8
// cells, 4 {cell, weight} words, or 4 weights with their 4 cells), the next runs'
// vectors being loaded before the current ones are added, and masks the elements
// outside the run.
//
// What bounds it: instructions and load latency.  On 12- or 8-byte records an
// event cost 1.35 (FP32) or about 1.2 (BF16) warp instructions; the split layouts
// move 2, 4 or 6 bytes an event, a 16-byte vector costs one load for 8 or 4 events,
// and an event costs 0.54 warp instructions and 2.2 bytes of DRAM with equal
// weights (1,314 spikes, 74 cells a run, 20.4 us cold at 37 % of the issue slots)
// and 0.76 and 4.2 as integers (2,400 spikes, 37 words, 24.6 us at 40 %).
//
// Accumulation is exact fixed point: a weight w becomes x = w 2^(q-s),
// split into hi = rint(x) and lo = rint((x - hi) 2^s) in [-2^(s-1), 2^(s-1)]
// (hi 2^s + lo = rint(w 2^q)); hi and lo are summed in two int32 arrays
// with shared-memory integer atomics, so the sum is order-independent and
// the cell value is (H 2^s + L) 2^-q.  The scales come from bounds on one
// launch: a cell receives at most E = min(spikes x max synapse
// multiplicity, max in-degree x spikes per neuron per interval) events of
// magnitude <= max|w|; s makes E 2^s < 2^31 and q makes
// E max|w| 2^(q-s) + E < 2^31, so neither sum can overflow, and the
// rounding error (<= 2^-(q+1) per event) is below that of FP32
// accumulation.  If no such scales exist the events are added in FP32 by
// shared-memory atomics.
//
// Uniform weights (kLayHom): a cell's sum is n0 w0 + n1 w1, so only the two
// counts are accumulated, in the halves of one 32-bit word (E <= 65,535; one
// addition of a constant per event, no weight to split), and the flush forms
// the same hi and lo sums from them.  Beyond that a two-word cell holds a count
// in each word, a one-word cell the sum of the integer weights (AddMode): 12,000
// spikes on 112,500 neurons, 346 (FP32) and 311 us (BF16) on whole records, 162
// and 156 so.
//
// The CTA then adds its cells into the ring buffer with fire-and-forget
// reductions: no other CTA touches them.  An external list whose emission
// steps span more than the window is delivered by the same CTAs with global
// atomics instead.
// ---------------------------------------------------------------------------
constexpr int kTileThreads = 1024;
constexpr int kTileWarps = kTileThreads / 32;

// One lane's vector of a run's stream.
template <int LAY> struct Vec { uint4 a; };
template <> struct Vec<kLayF32> {
  uint4 a;  // weights
  uint2 c;  // cells
};
template <int LAY> struct Lay {
  static constexpr uint32_t kElems = LAY == kLayHom ? 8u : 4u;
};
constexpr int kAhead = 3;  // vectors of a lane loaded ahead, for each of two runs
// Weight of element k of a vector.
template <int LAY>
__device__ __forceinline__ float vec_weight(const Vec<LAY>& x, int k) {
  const uint32_t w = k == 0 ? x.a.x : k == 1 ? x.a.y : k == 2 ? x.a.z : x.a.w;
  return __uint_as_float(LAY == kLayJ16 ? w & 0xFFFF0000u : w);
}

// One element of the stream, index i: its cell and its weight's bits.
template <int LAY> struct Elem { uint32_t a; };
template <> struct Elem<kLayF32> { uint32_t a, c; };
template <int LAY>
__device__ __forceinline__ Elem<LAY> load_elem(const NetView& v, uint64_t i) {
  Elem<LAY> x;
  if constexpr (LAY == kLayHom)
    x.a = __ldcs(reinterpret_cast<const uint16_t*>(v.dat) + i);
  else
    x.a = __ldcs(reinterpret_cast<const uint32_t*>(v.dat) + i);
  if constexpr (LAY == kLayF32) x.c = __ldcs(v.cells + i);
  return x;
}
template <int LAY>
__device__ __forceinline__ uint32_t elem_cell(const Elem<LAY>& x) {
  if constexpr (LAY == kLayF32) return x.c;
  else return x.a & 0xFFFFu;
}

__device__ __forceinline__ void red_shared_u32(uint32_t addr, uint32_t x) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
}
// The same where K < n (and, CLIP, K >= lo), else into the lane's own spare
// word `none`: a select (with the reduction under a condition an event took 1.25
// warp instructions in place of 0.8).
template <int K, bool CLIP>
__device__ __forceinline__ void red_shared_u32_at(uint32_t addr, uint32_t x,
                                                  int n, int lo, uint32_t none) {
  const bool on = CLIP ? (K < n && K >= lo) : K < n;
  red_shared_u32(on ? addr : none, x);
}

// base + 4 x the low (0) or high (1) half of w: one integer dot product.
template <int HALF>
__device__ __forceinline__ uint32_t cell_addr(uint32_t w, uint32_t base) {
  return __dp2a_lo(w, HALF ? 0x0400u : 0x0004u, base);
}

// Per-spike run for this CTA's tile, in elements of the store's stream (dat):
// the address of its first vector with the elements to skip there in the low
// bits, its end in elements from that vector on (top bit: uniform weight
// class), and the offset of its cells in the accumulator,
// (t - base + d_base) TW (a list outside the window: t).  Plastic tiles read
// element by element: the index of the first one, and the length.
struct SegDesc {
  uint64_t beg;
  uint32_t len;
  int32_t off;
#if SNN_CHECK
  uint64_t tgt;  // index of the run's first target, in words of its array
#endif
};

// Fixed-point scales of one launch (see above); fixed = 0: use FP32.
struct FixScale {
  int fixed;
  int packed;      // uniform weights: the counts fit 16 bits
  int sh;          // s
  float scale_hs;  // 2^(q - s)
  float scale_s;   // 2^s
  float inv_q;     // 2^-q (q <= 123: a normal float)
  float scale_sq;  // 2^(s-q)
};

// 2^k from the exponent bits (k inside the normal range of the type), and
// floor(log2 x) of a positive normal double.
__device__ __forceinline__ float pow2f(int k) {
  return __int_as_float((k + 127) << 23);
}
__device__ __forceinline__ double pow2d(int k) {
  return __longlong_as_double((long long)(k + 1023) << 52);
}
__device__ __forceinline__ int ilog2d(double x) {
  return (int)((__double_as_longlong(x) >> 52) & 0x7FF) - 1023;
}

// Largest s <= 23 and q - s <= 21 - ceil(log2 max|w|): a scaled weight
// x = w 2^(q-s) then has |x| < 2^22 and |(x - rint x) 2^s| <= 2^22, the
// range in which adding 1.5 2^23 rounds to an integer (fixed_split).
constexpr int kFixMaxShift = 23;

// Most events of a cell: a list of n_sp spikes, of one interval or of any steps.
__host__ __device__ inline uint64_t cell_events(const NetView& v, uint64_t n_sp,
                                                bool per_interval) {
  const uint64_t e = n_sp * (uint64_t)(v.mult_max ? v.mult_max : 1u);
  const uint64_t e2 = (uint64_t)v.k_in_max * (v.spikes_per_iv ? v.spikes_per_iv : 1u);
  return per_interval && e2 < e ? e2 : e;
}

__device__ FixScale fix_scale(const NetView& v, uint64_t n_sp,
                              bool per_interval) {
  FixScale f{0, 0, 0, 1.f, 1.f, 1.f, 1.f};
  const uint64_t e = cell_events(v, n_sp, per_interval);
  f.packed = e <= 0xFFFFull;
  if (e == 0 || e >= (1ull << 30) || !(v.max_abs_w > 0.f) ||
      !(v.max_abs_w <= 3.0e38f))
    return f;
  const int lg = 63 - __clzll((long long)e);  // 2^lg <= e < 2^(lg+1)
  const int sh = min(30 - lg, kFixMaxShift);  // e 2^sh < 2^31
  // largest qs with e max|w| 2^qs <= 2^31 - 1 - e: the hi sums (each
  // |hi| <= |x| + 1/2) cannot overflow
  const double A = 2147483647.0 - (double)e;
  const double B = (double)e * (double)v.max_abs_w;
  int qs = ilog2d(A) - ilog2d(B);  // floor(log2(A / B)) is qs or qs - 1
  if (B * pow2d(qs) > A) --qs;
  const uint32_t wb = __float_as_uint(v.max_abs_w);
  const int wexp = (int)((wb >> 23) & 0xFFu) - 127 + ((wb & 0x7FFFFFu) ? 1 : 0);
  qs = min(qs, 21 - wexp);
  if (qs < 0) return f;
  qs = min(qs, 100);
  // one-word cells hold hi only: lo must be zero for every weight
  if (v.acc_words == 1 && qs < v.acc_qs_min) return f;
  // (integer weights: the store's own scale, at most the launch's)
  if (v.lay == kLayI16) qs = v.acc_qs_min;
  const int q = sh + qs;
  f.fixed = 1;
  f.sh = sh;
  f.scale_hs = pow2f(qs);
  f.scale_s = pow2f(sh);
  f.inv_q = pow2f(-q);
  f.scale_sq = pow2f(-qs);
  return f;
}

// The two scales a split needs.
struct SplitScale {
  float scale_hs, scale_s;
};

// Exact split of x = w 2^(q-s) (|x| < 2^22, s <= 23): hi = rint(x),
// lo = rint((x - hi) 2^s), so hi 2^s + lo = rint(w 2^q).  Adding
// M = 1.5 2^23 puts a value of magnitude <= 2^22 into [2^23, 2^24], where
// the float spacing is 1: the sum is rounded to an integer (to nearest,
// ties to even) whose value is the bit pattern minus M's.  Only FMA-pipe
// arithmetic and integer subtractions; x (a product with a power of two) and
// x - hi are exact, so the fused forms round once, at the additions of M.
constexpr float kFixM = 12582912.0f;  // 1.5 * 2^23
template <class Scale>
__device__ __forceinline__ void fixed_split(float w, const Scale& fx,
                                            int& hi, int& lo) {
  const float y = __fmaf_rn(w, fx.scale_hs, kFixM);
  hi = __float_as_int(y) - __float_as_int(kFixM);
  const float fr = __fmaf_rn(w, fx.scale_hs, -__fsub_rn(y, kFixM));
  lo = __float_as_int(__fmaf_rn(fr, fx.scale_s, kFixM)) - __float_as_int(kFixM);
}

// Bounds-checked builds: a cell outside the store's window or one that
// disagrees with the synapse's target is skipped and flagged; so are targets
// outside the tile.  Production builds compile this to `true`.
[[maybe_unused]] __device__ __forceinline__ bool cell_in_bounds(const NetView& v, uint32_t cell,
                                               uint32_t tgt, uint32_t tgt_lo) {
  if (!kChecked) return true;
  const uint32_t d = cell / v.tile_w, j = cell - d * v.tile_w;
  const bool ok = tgt < v.n && tgt == tgt_lo + j &&
                  d + (uint32_t)v.d_base >= (uint32_t)v.d_min &&
                  d + (uint32_t)v.d_base <= (uint32_t)v.d_max;
  if (!ok) atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_CHECK);
  return ok;
}

// Plastic weight of an E->E synapse at its presynaptic spike t with delay
// d (pair-based power-law STDP, all pairs, the whole delay dendritic): the
// potentiation owed to the post spikes seen since the previous pre spike,
// in time order, then the depression by the post trace at t; weights stay in
// [0, w_max].  tprev / kprev: the previous pre spike and the presynaptic
// trace right after it.  The post spikes of target j come from the CTA's
// copy of its last hist spike times (rt: [hist][TW]; n: spikes so far); km
// is its post trace at t - d (from the CTA's table).
// Compiled once (not inlined into every unrolled record slot: the code would
// no longer fit the instruction cache).  .trunc = 1 when the potentiation
// window reached past the kept spikes.
struct StdpConst {
  float c_pot, c_dep, mu, w_max, l2_plus, l2_minus;
  uint32_t hmask;
};
struct StdpOut {
  float w;
  uint32_t trunc;
};

__device__ __noinline__ StdpOut stdp_weight(float w, int32_t t, uint32_t d,
                                            int32_t tprev, float kprev,
                                            uint32_t j, uint32_t TW,
                                            const int32_t* rt, float km,
                                            uint32_t n, StdpConst c) {
  StdpOut o;
  o.trunc = 0u;
  if (tprev != kNoSpike) {
    // post spikes seen in (previous pre spike, t]: newest first to find
    // the window, then applied oldest first
    const uint32_t H = c.hmask + 1u;
    const int32_t horizon = t - (int32_t)d;
    const int32_t after = tprev - (int32_t)d;
    const int32_t k_min = n > H ? (int32_t)(n - H) : 0;
    int32_t k_hi = -1, k_lo = -1, k = (int32_t)n - 1;
    for (; k >= k_min; --k) {
      const int32_t tp = rt[((uint32_t)k & c.hmask) * TW + j];
      if (tp > horizon) continue;
      if (tp <= after) break;
      if (k_hi < 0) k_hi = k;
      k_lo = k;
    }
    o.trunc = (k < k_min && n > H) ? 1u : 0u;
    if (k_lo >= 0) {
      // Where every power of two is a normal float the PTX instruction serves
      // (see ex2_normal): the longest lag of the window is t - tprev, and a
      // weight above 1e-30 stays above it (potentiation raises it, up to w_max),
      // so that mu log2 w >= -100 (mu <= 1).  112,500 neurons BF16 with STDP:
      // 8.6 ms a pass, 9.1 with exp2f alone.
      if (w > 1e-30f && c.w_max > 1e-30f &&
          (float)(t - tprev) * c.l2_plus <= 125.f) {
        for (int32_t q = k_lo; q <= k_hi; ++q) {
          const int32_t tp = rt[((uint32_t)q & c.hmask) * TW + j];
          const float kp = kprev * ex2_normal(-(float)(tp + (int32_t)d - tprev) * c.l2_plus);
          const float wm = ex2_normal(c.mu * log2f(w));
          w = fminf(w + c.c_pot * wm * kp, c.w_max);
        }
      } else {
        for (int32_t q = k_lo; q <= k_hi; ++q) {
          const int32_t tp = rt[((uint32_t)q & c.hmask) * TW + j];
          const float kp =
              kprev * exp2f(-(float)(tp + (int32_t)d - tprev) * c.l2_plus);
          const float wm = w > 0.f ? exp2f(c.mu * log2f(w)) : 0.f;
          w = fminf(w + c.c_pot * wm * kp, c.w_max);
        }
      }
    }
  }
  // depression by the post trace at t (from the CTA's table)
  o.w = fmaxf(w - c.c_dep * w * km, 0.f);
  return o;
}

// Where a tiled delivery's list comes from: the interval's own list, the
// partitions' exchange buffers (v.gx), a caller's arrays as they stand (v.ext_*),
// or a caller's list prepared in the own list's form (its steps: ext_tmin to
// ext_tmax of the control block).
enum ListKind { kListOwn, kListGathered, kListRaw, kListRange };
// A caller's list up to this long is read by every CTA as it stands (four
// entries a thread); a longer one is prepared by k_prepare_external first.
constexpr uint32_t kRawMax = 4 * kTileThreads;

// Places the run of elements [first, first + len) of v's stream in a
// descriptor.
template <int LAY>
__device__ __forceinline__ void place_run(const NetView& v, uint64_t first,
                                          uint32_t len, SegDesc* sd) {
  constexpr uint32_t E = Lay<LAY>::kElems;
  const uint32_t head = (uint32_t)first & (E - 1u);
  sd->beg = (reinterpret_cast<uint64_t>(v.dat) + (first / E) * 16u) | head;
  sd->len = len ? head + len : 0u;
}

// The launch's list as a delivery sees it: its length, the window's base
// step, whether its steps lie inside the window, and the clock.
struct ListView {
  uint32_t n_sp;
  bool inwin;
  long long base, t_now;
};

// Descriptors of the runs of spikes [j0, j0 + nb) for this CTA's tile: DU
// list entries per thread in flight, then their tile-index words and row
// starts.  pre (pre_g): entries threadIdx.x + u blockDim.x of the list, read
// ahead of its length (have_pre).  Returns the events described (gathered
// lists and callers' arrays).  wide: cells between the two populations' counts of
// a uniform store (0: halves of one word).  PL: also the presynaptic history the
// plastic rule needs.
template <int LAY, int DU, bool PL, int KIND>
__device__ __forceinline__ unsigned long long describe_runs(
    const NetView& v, const ListView& lv, const SpikeEntry* list, uint32_t tile,
    uint32_t j0, uint32_t nb, bool have_pre, const SpikeEntry* pre,
    const uint2* pre_g, const uint32_t* s_gstart, SegDesc* s_desc,
    uint32_t wide, int32_t* s_tprev, float* s_kprev, uint32_t* s_at) {
  constexpr bool GX = KIND == kListGathered, RAW = KIND == kListRaw;
  const uint32_t row_stride = v.n_tiles + 1;
  const uint32_t iv_span = (uint32_t)(v.window - (v.d_max - v.d_min));
  unsigned long long my_events = 0;
  for (uint32_t k0 = threadIdx.x; k0 < nb; k0 += DU * blockDim.x) {
    uint32_t src[DU];
    int32_t t[DU];
    const bool have = have_pre && j0 == 0 && k0 == threadIdx.x;
#pragma unroll
    for (int u = 0; u < DU; ++u) {
      const uint32_t k = k0 + u * blockDim.x;
      src[u] = 0xFFFFFFFFu;
      t[u] = 0;
      if (k < nb) {
        if constexpr (GX) {
          const uint32_t g = j0 + k;
          uint32_t p = 0;
          while (s_gstart[p + 1] <= g) ++p;
          const uint2 x = (have && p == 0)
              ? pre_g[u]
              : reinterpret_cast<const uint2*>(
                    v.gx + (uint64_t)p * v.gx_stride + 4)[g - s_gstart[p]];
          // entries come from the caller's buffers: a source outside the
          // store or a step outside this interval is skipped and flagged
          // (its cells would lie outside the tile's window)
          const bool ok = x.x < v.n_src &&
                          (uint32_t)((int32_t)x.y - (int32_t)lv.t_now) < iv_span;
          if (!ok) atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_BAD_SOURCE);
          src[u] = ok ? x.x : 0xFFFFFFFFu;
          t[u] = (int32_t)x.y;
        } else if constexpr (RAW) {
          const uint2 x = have ? pre_g[u]
                               : make_uint2(v.ext_src[j0 + k], (uint32_t)v.ext_t[j0 + k]);
          if (x.x >= v.n_src) atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_BAD_SOURCE);
          src[u] = x.x;
          t[u] = (int32_t)x.y;
        } else {
          const SpikeEntry e = have ? pre[u] : list[j0 + k];
          src[u] = e.src;
          t[u] = e.t;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < DU; ++u) {
      const uint32_t k = k0 + u * blockDim.x;
      if (k >= nb) continue;
      SegDesc sd{};
      sd.off = lv.inwin ? (int32_t)((long long)t[u] - lv.base + v.d_base) *
                              (int32_t)v.tile_w
                        : t[u];
      if (src[u] < v.n_src) {
        const uint32_t* to = v.tile_off + (uint64_t)src[u] * row_stride + tile;
        const uint32_t a = to[0], b = to[1];
        const uint64_t row = v.row_ptr[src[u]];
        uint32_t len = b - a;
#if SNN_CHECK
        const uint64_t row_end = v.row_ptr[src[u] + 1];
        sd.tgt = v.fmt == SNN_W_FP32_12B ? row + a
                                         : 2 * row + (row_end - row) + a;
        if (b < a || row + b > row_end) {
          atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_CHECK);
          len = 0;
        }
#endif
        if (GX || RAW) my_events += len;
        if constexpr (PL) {
          sd.beg = row * v.row_mul + a;
          sd.len = len;
          s_at[k] = a;
        } else {
          place_run<LAY>(v, row * v.row_mul + a, len, &sd);
          // (counts in words of their own: the second population's further on)
          if (LAY == kLayHom && src[u] >= v.hom_split) {
            if (wide) sd.off += (int32_t)wide;
            else sd.len |= 0x80000000u;
          }
        }
      }
      s_desc[k] = sd;
      if constexpr (PL) {
        const bool exc = src[u] < v.sp.n_exc;
        s_tprev[k] = exc ? v.sp.prev_t[src[u]] : kNoSpike;
        s_kprev[k] = exc ? v.sp.prev_k[src[u]] : -1.f;
      }
    }
  }
  // the warp's events (all threads of the CTA reach this)
  if (GX || RAW) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) my_events += __shfl_xor_sync(kFull, my_events, o);
  }
  return my_events;
}

// Value of one accumulator cell, the FP32 sum of its events: exact sums
// (H 2^s + L) 2^-q as H 2^(s-q) + L 2^-q (both products are exact while |H|
// and |L| are below 2^24 -- then only the addition rounds, so the result is
// the correctly rounded sum; larger words round once more; no 64-bit
// conversion or FP64 arithmetic, whose rate is low on this part).  Uniform
// weights: H and L from the two counts of the cell.
enum CellKind { kCellFloat, kCellOne, kCellTwo, kCellCounts, kCellCountsOne,
                kCellCountsFloat, kCellWide, kCellWideFloat };
struct CellValue {
  float scale_sq, inv_q;
  int h0, l0, h1, l1;
  float w0, w1;
  __device__ __forceinline__ CellValue(const NetView& v, const FixScale& f)
      : scale_sq(f.scale_sq), inv_q(f.inv_q), h0(0), l0(0), h1(0), l1(0),
        w0(v.hom_w[0]), w1(v.hom_w[1]) {
    if (v.lay == kLayHom && f.fixed) {
      fixed_split(w0, f, h0, l0);
      fixed_split(w1, f, h1, l1);
    }
  }
  // c: the cell's index; cells: the accumulator's
  template <int KIND>
  __device__ __forceinline__ float get(const int* acc, uint32_t c,
                                       uint32_t cells) const {
    int H = acc[c], L = 0;
    if (KIND == kCellFloat) return __int_as_float(H);
    if (KIND >= kCellCounts) {
      constexpr bool WIDE = KIND == kCellWide || KIND == kCellWideFloat;
      const int n0 = WIDE ? H : H & 0xFFFF;
      const int n1 = WIDE ? acc[cells + c] : (int)((uint32_t)H >> 16);
      if (KIND == kCellCountsFloat || KIND == kCellWideFloat) {
        // (a count of zero adds nothing, also where the weight is infinite)
        const float b = n1 ? __fmul_rn((float)n1, w1) : 0.f;
        return n0 ? __fmaf_rn((float)n0, w0, b) : b;
      }
      H = n0 * h0 + n1 * h1;
      L = n0 * l0 + n1 * l1;
    } else if (KIND == kCellTwo) {
      L = acc[cells + c];
    }
    float a = __fmul_rn(__int2float_rn(H), scale_sq);
    if (KIND == kCellTwo || KIND == kCellCounts || KIND == kCellWide)
      a = __fadd_rn(a, __fmul_rn(__int2float_rn(L), inv_q));
    return a;
  }
};

// Adds the tile's window into the ring buffer: every cell belongs to this CTA
// alone, so its sum goes out as a fire-and-forget global reduction: the one
// addition rb + sum that a read-modify-write would make, without a memory
// round trip (the slots of a column are independent: unrolled, so that their
// shared-memory reads and conversions overlap).
template <int KIND>
__device__ __forceinline__ void flush_kind(const NetView& v, const CellValue& val,
                                           const int* acc, uint32_t tgt_lo,
                                           long long base) {
  const uint32_t TW = v.tile_w, W = (uint32_t)v.window, cells = W * TW;
  const uint32_t x_end = tgt_lo < v.n ? min(TW, v.n - tgt_lo) : 0u;
  for (uint32_t x = threadIdx.x; x < x_end; x += blockDim.x) {
    float* const col = v.rb + tgt_lo + x;
#pragma unroll 4
    for (uint32_t sl = 0; sl < W; ++sl) {
      const float a = val.get<KIND>(acc, sl * TW + x, cells);
      if (a != 0.f)
        red_add_f32(col + (size_t)((uint32_t)(base + sl) & v.slot_mask) * v.pitch, a);
    }
  }
}
template <bool HOM, bool WIDE>
__device__ __forceinline__ void flush_tile(const NetView& v, const FixScale& fx,
                                           bool two, const int* acc,
                                           uint32_t tgt_lo, long long base) {
  const CellValue val(v, fx);
  if (WIDE) {
    if (!fx.fixed) flush_kind<kCellWideFloat>(v, val, acc, tgt_lo, base);
    else flush_kind<kCellWide>(v, val, acc, tgt_lo, base);
  } else if (HOM && fx.packed) {
    if (!fx.fixed) flush_kind<kCellCountsFloat>(v, val, acc, tgt_lo, base);
    else if (two) flush_kind<kCellCounts>(v, val, acc, tgt_lo, base);
    else flush_kind<kCellCountsOne>(v, val, acc, tgt_lo, base);
  } else if (!fx.fixed) {
    flush_kind<kCellFloat>(v, val, acc, tgt_lo, base);
  } else if (two) {
    flush_kind<kCellTwo>(v, val, acc, tgt_lo, base);
  } else {
    flush_kind<kCellOne>(v, val, acc, tgt_lo, base);
  }
}

// A CTA's end of a list: the last of the list's CTAs clears its counters and,
// for the interval's own list, commits its events and advances the clock.
__device__ __forceinline__ void finish_list(const NetView& v,
                                            unsigned long long* pair_p,
                                            unsigned int* done_p,
                                            int advance_time, bool gathered) {
  __threadfence();
  const unsigned prev = atomicAdd(done_p, 1u);
  if (prev != v.n_tiles - 1) return;
  *pair_p = 0ull;
  *done_p = 0u;
  if (!advance_time) return;
  // this net's exchange list has been read (by the collective before this
  // delivery, or by this delivery itself): the next update refills it
  if (v.xbuf) *v.xbuf = 0u;
  v.ctl->t_now += v.ctl->iv_steps;
  const unsigned long long own = atomicExch(&v.ctl->pending_events, 0ull);
  v.ctl->events += gathered ? atomicExch(&v.ctl->gx_events, 0ull) : own;
}

// The events of one vector: elements K of [lo, n) (CLIP; else [0, n)).
template <int LAY, bool CLIP, int K>
__device__ __forceinline__ void add_elem(const Vec<LAY>& x, uint32_t row_s,
                                         uint32_t inc, int n, int lo,
                                         uint32_t lo_off, uint32_t none,
                                        const SplitScale& fx) {
  if constexpr (LAY == kLayHom) {
    const uint32_t w = K < 2 ? x.a.x : K < 4 ? x.a.y : K < 6 ? x.a.z : x.a.w;
    red_shared_u32_at<K, CLIP>(cell_addr<K & 1>(w, row_s), inc, n, lo, none);
  } else if constexpr (LAY == kLayI16) {
    const uint32_t w = K == 0 ? x.a.x : K == 1 ? x.a.y : K == 2 ? x.a.z : x.a.w;
    red_shared_u32_at<K, CLIP>(cell_addr<0>(w, row_s), (uint32_t)((int)w >> 16), n, lo,
                               none);
  } else {
    uint32_t addr;
    if constexpr (LAY == kLayF32)
      addr = cell_addr<K & 1>(K < 2 ? x.c.x : x.c.y, row_s);
    else
      addr = cell_addr<0>(K == 0 ? x.a.x : K == 1 ? x.a.y : K == 2 ? x.a.z : x.a.w, row_s);
    int hi, low;
    fixed_split(vec_weight<LAY>(x, K), fx, hi, low);
    red_shared_u32_at<K, CLIP>(addr, (uint32_t)hi, n, lo, none);
    // (one-word cells have no low part)
    red_shared_u32_at<K, CLIP>(LAY == kLayF32 || lo_off ? addr + lo_off : none,
                               (uint32_t)low, n, lo, none);
  }
}
template <int LAY, bool CLIP>
__device__ __forceinline__ void add_vec(const Vec<LAY>& x, uint32_t row_s,
                                        uint32_t inc, int n, int lo,
                                        uint32_t lo_off, uint32_t none,
                                        const SplitScale& fx) {
  add_elem<LAY, CLIP, 0>(x, row_s, inc, n, lo, lo_off, none, fx);
  add_elem<LAY, CLIP, 1>(x, row_s, inc, n, lo, lo_off, none, fx);
  add_elem<LAY, CLIP, 2>(x, row_s, inc, n, lo, lo_off, none, fx);
  add_elem<LAY, CLIP, 3>(x, row_s, inc, n, lo, lo_off, none, fx);
  if constexpr (Lay<LAY>::kElems == 8) {
    add_elem<LAY, CLIP, 4>(x, row_s, inc, n, lo, lo_off, none, fx);
    add_elem<LAY, CLIP, 5>(x, row_s, inc, n, lo, lo_off, none, fx);
    add_elem<LAY, CLIP, 6>(x, row_s, inc, n, lo, lo_off, none, fx);
    add_elem<LAY, CLIP, 7>(x, row_s, inc, n, lo, lo_off, none, fx);
  }
}

// A lane's part of one run: its first vectors, the elements of the run from
// the first of them on (n; those before `lo` belong to the row's previous
// run), the run's cells in the accumulator and its increment.
template <int LAY> struct LaneRun {
  Vec<LAY> x[kAhead];
  const char* p;   // the lane's first vector
  int n, lo;
  uint32_t row_s, inc;
#if SNN_CHECK
  uint64_t tgt;    // index of the target of the lane's element 0
  int32_t off;
#endif
};

// Bounds-checked builds: what the vectors and elements of a tile's runs are
// checked against; the vector at p must lie in the store, an element's cell in
// its window, on its target and in the accumulator.
#if SNN_CHECK
struct RunCheck {
  const NetView* v;
  uint32_t tgt_lo;
  uint32_t acc_len;  // cells of the accumulator
};
__device__ __forceinline__ bool flag_check(const NetView& v, bool ok) {
  if (!ok) atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_CHECK);
  return ok;
}
__device__ __forceinline__ bool vec_in_store(const NetView& v, const char* p) {
  const uint64_t b = reinterpret_cast<uint64_t>(p) - reinterpret_cast<uint64_t>(v.dat);
  const uint64_t bytes =
      v.fmt != SNN_W_FP32_12B ? 8 * v.n_pad : (v.lay == kLayHom ? 2 : 4) * v.n_pad;
  return flag_check(v, b % 16 == 0 && b < bytes && b + 16 <= bytes);
}
template <int LAY>
__device__ __forceinline__ uint32_t vec_cell(const Vec<LAY>& x, int k) {
  uint32_t w;
  if constexpr (LAY == kLayF32) w = k < 2 ? x.c.x : x.c.y;
  else if constexpr (LAY == kLayHom)
    w = k < 2 ? x.a.x : k < 4 ? x.a.y : k < 6 ? x.a.z : x.a.w;
  else w = k == 0 ? x.a.x : k == 1 ? x.a.y : k == 2 ? x.a.z : x.a.w;
  return (LAY == kLayF32 || LAY == kLayHom) && (k & 1) ? w >> 16 : w & 0xFFFFu;
}
#define SNN_CHECKED(...) , __VA_ARGS__
#else
#define SNN_CHECKED(...)
#endif

// Phase (B) for a batch of nb described runs, 2^lg lanes a run: every warp
// takes each kTileWarps-th group of 32 / 2^lg runs, and loads a lane's first
// kAhead vectors of the next group before it adds the current one.
// (Measured and not kept: masks only on a run's first and last vector, held
// apart from the whole ones -- a fifth fewer instructions, but more registers
// and branches: 29.8 -> 34.9 us on the 112,500-neuron list.)
// inc0, inc1: what an event of uniform weight adds, by population.
template <int LAY>
__device__ __forceinline__ void add_runs(const char* dat, const char* cel,
                                      const SegDesc* s_desc, uint32_t nb,
                                      uint32_t acc_s, uint32_t lo_off,
                                      uint32_t lg,
                                      SplitScale fx SNN_CHECKED(RunCheck chk),
                                      uint32_t inc0 = 1u, uint32_t inc1 = 0x10000u) {
  constexpr uint32_t E = Lay<LAY>::kElems;
  __shared__ uint32_t s_none[32];  // what masked elements add to
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t none = (uint32_t)__cvta_generic_to_shared(s_none + lane);
  const uint32_t L = 1u << lg, R = 32u >> lg;
  const int kStep = (int)(L * E);  // elements between a lane's vectors
  const uint32_t sub = lane & (L - 1u);
  const uint32_t stride = kTileWarps * R;
  // (FP32 weights at dat: their cells, half the bytes, at cel)
  auto fetch = [&](const LaneRun<LAY>& r, int q) {
    const char* p = r.p + (size_t)q * (L * 16u);
    Vec<LAY> x;
    x.a = __ldcs(reinterpret_cast<const uint4*>(p));
    if constexpr (LAY == kLayF32)
      x.c = __ldcs(reinterpret_cast<const uint2*>(cel + ((p - dat) >> 1)));
    return x;
  };
  auto load = [&](LaneRun<LAY>& r, uint32_t j) {
    r.n = 0;
    if (j < nb) {
      const SegDesc sd = s_desc[j];
      r.p = reinterpret_cast<const char*>((sd.beg & ~15ull) + sub * 16u);
      r.lo = sub == 0 ? (int)((uint32_t)sd.beg & 15u) : 0;
      r.n = (int)(sd.len & 0x7FFFFFFFu) - (int)(sub * E);
      r.row_s = acc_s + 4u * (uint32_t)sd.off;
      r.inc = (int)sd.len < 0 ? inc1 : inc0;
#if SNN_CHECK
      r.tgt = sd.tgt + sub * E - (sd.beg & 15u);
      r.off = sd.off;
      for (int q = 0; r.n > q * kStep; ++q)
        if (!vec_in_store(*chk.v, r.p + (size_t)q * (L * 16u))) r.n = q * kStep;
#endif
#pragma unroll
      for (int q = 0; q < kAhead; ++q)
        if (r.n > q * kStep) r.x[q] = fetch(r, q);
    }
  };
  // elements [lo, r.n - q kStep) of the lane's vector q; CLIP: lo may not be 0
  auto put = [&](auto clip, const LaneRun<LAY>& r, const Vec<LAY>& x, int q, int lo) {
    constexpr bool CLIP = decltype(clip)::value;
    const int n = r.n - q * kStep;
#if SNN_CHECK
    uint32_t good = 0, all = 0;
    for (int k = lo; k < min(n, (int)E); ++k) {
      const uint32_t cell = vec_cell<LAY>(x, k);
      const uint64_t ti = r.tgt + (uint64_t)(q * kStep + k);
      const uint32_t tgt = chk.v->tgts ? chk.v->tgts[ti]
                                       : reinterpret_cast<const uint32_t*>(chk.v->recs)[ti];
      all |= 1u << k;
      if (cell_in_bounds(*chk.v, cell, tgt, chk.tgt_lo) &&
          flag_check(*chk.v, (uint32_t)r.off + cell < chk.acc_len))
        good |= 1u << k;
    }
    if (good != all) {  // the others one by one
      for (int k = 0; k < (int)E; ++k)
        if (good >> k & 1u)
          add_vec<LAY, true>(x, r.row_s, r.inc, k + 1, k, lo_off, none, fx);
      return;
    }
#endif
    add_vec<LAY, CLIP>(x, r.row_s, r.inc, n, lo, lo_off, none, fx);
  };
  auto add = [&](LaneRun<LAY>& r) {
    if (r.n > 0) put(std::true_type{}, r, r.x[0], 0, r.lo);
#pragma unroll
    for (int q = 1; q < kAhead; ++q)
      if (r.n > q * kStep) put(std::false_type{}, r, r.x[q], q, 0);
    for (int q = kAhead; r.n > q * kStep; ++q) {
      const Vec<LAY> x = fetch(r, q);
      put(std::false_type{}, r, x, q, 0);
    }
  };
  uint32_t k = (threadIdx.x >> 5) * R;
  const uint32_t grp = lane >> lg;
  LaneRun<LAY> a, b;
  load(a, k + grp);
  for (; k < nb; k += 2 * stride) {
    load(b, k + stride + grp);
    add(a);
    load(a, k + 2 * stride + grp);
    add(b);
  }
}

// The same out of line, for a kernel whose own registers it would not fit
// beside.
template <int LAY>
__device__ __noinline__ void add_runs_call(const char* dat, const char* cel,
                                           const SegDesc* s_desc, uint32_t nb,
                                           uint32_t acc_s, uint32_t lo_off,
                                           uint32_t lg,
                                           SplitScale fx SNN_CHECKED(RunCheck chk)) {
  add_runs<LAY>(dat, cel, s_desc, nb, acc_s, lo_off, lg, fx SNN_CHECKED(chk));
}

template <int LAY, int KIND>
__device__ __forceinline__ void deliver_tile_outside(
    const NetView& v, unsigned long long* pair_p, unsigned int* done_p,
    const SpikeEntry* __restrict__ list, uint32_t tile, int* acc_mem,
    uint32_t desc_off, uint32_t desc_cap);

// One interval's (or one caller's) list for tile `tile`.
template <int LAY, bool COUNT, int KIND, int MODE>
__device__ __forceinline__ void deliver_tile_body(
    const NetView& v, unsigned long long* pair_p, unsigned int* done_p,
    const SpikeEntry* __restrict__ list, int advance_time,
    uint32_t tile, int* acc_mem, uint32_t desc_off, uint32_t desc_cap) {
  static_assert(MODE == kAddAny || !COUNT, "counted cells are added one by one");
  static_assert((MODE != kAddWeighted && MODE != kAddWide) || LAY == kLayHom,
                "uniform weights");
  constexpr bool GX = KIND == kListGathered, RAW = KIND == kListRaw;
  constexpr bool RANGE = KIND == kListRange;
  SegDesc* const s_desc =
      reinterpret_cast<SegDesc*>(reinterpret_cast<char*>(acc_mem) + desc_off);
  __shared__ FixScale s_fx;
  __shared__ int s_range[2];  // callers' arrays: first and last emission step
  __shared__ uint32_t s_gstart[GX ? kMaxGatherParts + 1 : 1];
  __shared__ unsigned long long s_events;  // (GX, RAW) this CTA's events
  const uint32_t TW = v.tile_w;
  const uint32_t W = (uint32_t)v.window;
  const uint32_t cells = W * TW;
  // hi and lo words per cell (FP32 weights' 24-bit significands never sit on
  // a grid as coarse as a launch's step)
  const bool two = LAY != kLayI16 && v.acc_words == 2;
  const uint32_t tgt_lo = tile * TW;
  const unsigned lane = threadIdx.x & 31u;
  // An interval's own list (capacity list_cap): this thread's first list
  // entries are read together with the list's length, not after it (one
  // memory round trip fewer before the runs can be described); entries past
  // the length are never used.
  constexpr int kDU = 4;
  SpikeEntry pre[GX || RAW ? 1 : kDU];
  uint2 pre_g[GX || RAW ? kDU : 1];
  constexpr bool spec = !RANGE;
  if constexpr (spec) {
#pragma unroll
    for (int u = 0; u < kDU; ++u) {
      const uint32_t k = threadIdx.x + u * blockDim.x;
      if constexpr (RAW) {
        pre_g[u] = make_uint2(0xFFFFFFFFu, 0u);
        if (k < v.ext_n) pre_g[u] = make_uint2(v.ext_src[k], (uint32_t)v.ext_t[k]);
      } else if constexpr (GX) {  // part 0's first entries (its count comes next)
        if (k < desc_cap && k < v.gx_cap)
          pre_g[u] = reinterpret_cast<const uint2*>(v.gx + 4)[k];
      } else {
        if (k < desc_cap && k < v.list_cap) pre[u] = list[k];
      }
    }
  }
  // every thread reads the launch's list size and window (same addresses); the
  // last one derives the fixed-point scales meanwhile
  ListView lv;
  if constexpr (GX) {
    // the parts' counts (each at most its capacity) and their starts in the
    // union, in part order; every thread computes them (same values, no
    // barrier) from the same words
    uint32_t run = 0;
    for (uint32_t p = 0; p < v.gx_parts; ++p) {
      s_gstart[p] = run;
      run += min(*reinterpret_cast<const volatile uint32_t*>(
                     v.gx + (uint64_t)p * v.gx_stride),
                 v.gx_cap);
    }
    s_gstart[v.gx_parts] = run;
    lv.n_sp = run;
  } else if constexpr (RAW) {
    lv.n_sp = v.ext_n;
    if (threadIdx.x == 0) {
      s_range[0] = INT_MAX;
      s_range[1] = INT_MIN;
      s_events = 0ull;
    }
    __syncthreads();
    int lo = INT_MAX, hi = INT_MIN;
#pragma unroll
    for (int u = 0; u < kDU; ++u)
      if (threadIdx.x + u * blockDim.x < v.ext_n) {
        lo = min(lo, (int)pre_g[u].y);
        hi = max(hi, (int)pre_g[u].y);
      }
    lo = __reduce_min_sync(kFull, lo);
    hi = __reduce_max_sync(kFull, hi);
    if (lane == 0 && lo <= hi) {
      atomicMin(&s_range[0], lo);
      atomicMax(&s_range[1], hi);
    }
    __syncthreads();
  } else {
    const unsigned long long pr =
        *reinterpret_cast<volatile unsigned long long*>(pair_p);
    lv.n_sp = (uint32_t)(pr >> 32);
  }
  lv.t_now = GX ? v.ctl->t_now : 0ll;
  if (RAW || RANGE) {
    const long long tmin = RAW ? s_range[0] : v.ctl->ext_tmin;
    const long long tmax = RAW ? s_range[1] : v.ctl->ext_tmax;
    lv.base = tmin + v.d_min;
    lv.inwin = (tmax - tmin) + (v.d_max - v.d_min) + 1 <= (long long)W;
  } else {
    lv.base = v.ctl->t_now + v.d_min;
    lv.inwin = true;
  }
  if constexpr (MODE != kAddAny && (RAW || RANGE)) {
    if (!lv.inwin) {  // (uniform: every thread has the same steps)
      deliver_tile_outside<LAY, KIND>(v, pair_p, done_p, list, tile, acc_mem,
                                      desc_off, desc_cap);
      return;
    }
  }
  const uint32_t n_sp = lv.n_sp;
  const long long base = lv.base;
  constexpr bool PER_IV = !RAW && !RANGE;
  // (the last thread: it describes no run of a list of up to 1,023 spikes)
  if (threadIdx.x == kTileThreads - 1) {
    const FixScale f = fix_scale(v, n_sp, PER_IV);
    s_fx = f;
    // (counts need no scales: weights that have none are added up as floats)
    if (MODE != kAddAny && n_sp &&
        !(MODE == kAddWide || (MODE == kAddVectors && LAY == kLayHom ? f.packed : f.fixed)))
      atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_SCALES);
  }
  if (GX && threadIdx.x == 0) s_events = 0ull;
  const bool one = MODE == kAddVectors && LAY == kLayHom ? true
                   : MODE == kAddWide                    ? false
                                                         : !two;
  for (uint32_t x = threadIdx.x; x < (one ? cells : 2 * cells); x += blockDim.x)
    acc_mem[x] = 0;
  const uint32_t acc_s = (uint32_t)__cvta_generic_to_shared(acc_mem);
  FixScale fx{};  // the last thread's s_fx, read after the first barrier

  // kAddAny: a list outside the window, no exact sums, counted cells.  2^lg lanes
  // take a run, a lane every 2^lg-th element, PER of each of a lane's U runs loaded
  // before any is added: where an event costs a global reduction, neighbouring
  // lanes' targets share L2 lines.  What bounds it there are those reductions
  // (2.6e11/s).  On whole records, with vectors of different runs on the lanes one
  // at a time and a division an event, and here: 12,000 spikes across 45 steps,
  // 112,500 neurons of equal weights 612, 752, 517 us, 50,021 neurons BF16 412, 449,
  // 397 us; 20 counted intervals of the former 2,487, 3,120, 2,237 us.
  [[maybe_unused]] auto add_any = [&](uint32_t nb) {
    constexpr int U = LAY == kLayF32 ? 2 : 4;
    constexpr int PER = 3;
    const uint32_t magic = cell_magic(TW);
    int h[2] = {0, 0}, l[2] = {0, 0};  // uniform weights
    if (LAY == kLayHom && fx.fixed) {
      fixed_split(v.hom_w[0], fx, h[0], l[0]);
      fixed_split(v.hom_w[1], fx, h[1], l[1]);
    }
    auto event = [&](const SegDesc& sd, const Elem<LAY>& x) {
      const uint32_t cell = elem_cell<LAY>(x);
      const bool c1 = (int)sd.len < 0;
      float w;
      if constexpr (LAY == kLayHom) w = c1 ? v.hom_w[1] : v.hom_w[0];
      else if constexpr (LAY == kLayI16) w = (float)((int)x.a >> 16) * pow2f(-v.acc_qs_min);
      else w = __uint_as_float(LAY == kLayF32 ? x.a : x.a & 0xFFFF0000u);
      if (lv.inwin) {
        const uint32_t c = (uint32_t)sd.off + cell;
        if (LAY == kLayHom && fx.packed) {
          red_shared_u32(acc_s + 4u * c, c1 ? 0x10000u : 1u);
        } else if (fx.fixed) {
          int hi, lo;
          if constexpr (LAY == kLayHom) {
            hi = c1 ? h[1] : h[0];
            lo = c1 ? l[1] : l[0];
          } else {
            fixed_split(w, fx, hi, lo);
          }
          red_shared_u32(acc_s + 4u * c, (uint32_t)hi);
          if (two && lo != 0) red_shared_u32(acc_s + 4u * (cells + c), (uint32_t)lo);
        } else {
          atomicAdd(reinterpret_cast<float*>(acc_mem) + c, w);
        }
        if (COUNT) {
          const uint32_t sl = cell_step(c, magic);
          atomicAdd(v.counts + (size_t)((uint32_t)(base + sl) & v.slot_mask) * v.pitch +
                        tgt_lo + (c - sl * TW), 1u);
        }
      } else {
        const uint32_t d = cell_step(cell, magic);
        const size_t at =
            (size_t)(((uint32_t)sd.off + d + (uint32_t)v.d_base) & v.slot_mask) * v.pitch +
            tgt_lo + (cell - d * TW);
        red_add_f32(v.rb + at, w);
        if (COUNT) atomicAdd(v.counts + at, 1u);
      }
    };
    // element idx of a run that starts at element i0 of the stream
    auto put = [&](const SegDesc& sd, uint32_t idx, const Elem<LAY>& x) {
#if SNN_CHECK
      const uint64_t ti = sd.tgt + idx;
      const uint32_t tgt = v.tgts ? v.tgts[ti]
                                  : reinterpret_cast<const uint32_t*>(v.recs)[ti];
      if (!cell_in_bounds(v, elem_cell<LAY>(x), tgt, tgt_lo)) return;
#endif
      event(sd, x);
    };
    auto first = [&](const SegDesc& sd) {
      return ((sd.beg & ~15ull) - reinterpret_cast<uint64_t>(v.dat)) / 16u *
                 Lay<LAY>::kElems + (sd.beg & 15u);
    };
    auto length = [&](const SegDesc& sd) {
      const uint32_t m = sd.len & 0x7FFFFFFFu;
      return m ? m - ((uint32_t)sd.beg & 15u) : 0u;
    };
    // lanes a run: three elements each for a mean run and a standard deviation
    const float run = v.mean_row / (float)v.n_tiles;
    uint32_t lg = 0;
    while (lg < 5u && ((nb << (lg + 1u)) <= (uint32_t)kTileThreads ||
                       3.f * (float)(1u << lg) < run + sqrtf(run)))
      ++lg;
    const uint32_t L = 1u << lg, R = 32u >> lg, sub = lane & (L - 1u);
    for (uint32_t k0 = (threadIdx.x >> 5) * U * R; k0 < nb; k0 += kTileWarps * U * R) {
      Elem<LAY> x[U][PER];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t j = k0 + u * R + (lane >> lg);
        if (j >= nb) continue;
        const SegDesc sd = s_desc[j];
        const uint64_t i0 = first(sd) + sub;
        const uint32_t len = length(sd);
#pragma unroll
        for (int q = 0; q < PER; ++q)
          if (sub + L * q < len) x[u][q] = load_elem<LAY>(v, i0 + L * q);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t j = k0 + u * R + (lane >> lg);
        if (j >= nb) continue;
        const SegDesc sd = s_desc[j];
        const uint32_t len = length(sd);
#pragma unroll
        for (int q = 0; q < PER; ++q)
          if (sub + L * q < len) put(sd, sub + L * q, x[u][q]);
        for (uint32_t idx = PER * L + sub; idx < len; idx += L)
          put(sd, idx, load_elem<LAY>(v, first(sd) + idx));
      }
    }
  };

  uint32_t j0 = 0;
  do {
    const uint32_t nb = min(desc_cap, n_sp - j0);
    const unsigned long long warp_events = describe_runs<LAY, kDU, false, KIND>(
        v, lv, list, tile, j0, nb, spec, pre, pre_g, s_gstart, s_desc,
        MODE == kAddWide ? cells : 0u, nullptr, nullptr, nullptr);
    // a batch of few runs spreads them over all lanes of the CTA
    uint32_t lg = (uint32_t)v.lg;
    while (lg < 5u && (nb << (lg + 1u)) <= (uint32_t)kTileThreads) ++lg;
    __syncthreads();
    // (after the barrier: s_events was cleared before it)
    if ((GX || RAW) && lane == 0 && warp_events) atomicAdd(&s_events, warp_events);
    fx = s_fx;
#if SNN_CHECK
    const RunCheck chk{&v, tgt_lo, MODE == kAddWide ? 2 * cells : cells};
#endif
    if constexpr (MODE == kAddAny) {
      add_any(nb);
    } else if constexpr (MODE == kAddWeighted) {
      int h[2], l;
      fixed_split(v.hom_w[0], fx, h[0], l);
      fixed_split(v.hom_w[1], fx, h[1], l);
      add_runs<LAY>(reinterpret_cast<const char*>(v.dat), nullptr, s_desc, nb, acc_s, 0u,
                    lg, SplitScale{} SNN_CHECKED(chk), (uint32_t)h[0], (uint32_t)h[1]);
    } else {
      add_runs<LAY>(reinterpret_cast<const char*>(v.dat),
                    reinterpret_cast<const char*>(v.cells), s_desc, nb, acc_s,
                    two ? 4u * cells : 0u, lg,
                    SplitScale{fx.scale_hs, fx.scale_s} SNN_CHECKED(chk));
    }
    j0 += nb;
    __syncthreads();  // s_desc is rewritten by the next batch
  } while (j0 < n_sp);
  if (lv.inwin)
    flush_tile<LAY == kLayHom && MODE != kAddWeighted, MODE == kAddWide>(v, fx, two, acc_mem,
                                                                         tgt_lo, base);
  // The last CTA to finish clears the list counters and advances the clock
  // (a gathered list's events -- its spikes' runs onto this partition's
  // targets -- are counted by the CTAs themselves).
  // A caller's arrays leave no counters behind but the events.
  __syncthreads();
  if (threadIdx.x == 0) {
    if (RAW) {
      if (s_events) atomicAdd(&v.ctl->events, s_events);
    } else {
      if (GX && s_events) atomicAdd(&v.ctl->gx_events, s_events);
      finish_list(v, pair_p, done_p, advance_time, GX);
    }
  }
}

// The same for a plastic net's tile (snn_set_stdp): E->E events apply the
// weight rule to their FP32 weight first.  A warp takes U runs at a time,
// three records per lane of each loaded before any is added (the rule's
// registers leave no room for more), in fixed shares: the plastic net's own
// lists are always inside the window.
template <int LAY, bool COUNT>
__device__ __forceinline__ void deliver_tile_plastic(
    const NetView& v, unsigned long long* pair_p, unsigned int* done_p,
    const SpikeEntry* __restrict__ list, int advance_time, uint32_t tile,
    int* acc_mem, uint32_t desc_off, uint32_t desc_cap) {
  constexpr int U = LAY == kLayF32 ? 1 : 2;
  constexpr int PER = 3;
  SegDesc* const s_desc =
      reinterpret_cast<SegDesc*>(reinterpret_cast<char*>(acc_mem) + desc_off);
  int32_t* const s_tprev = reinterpret_cast<int32_t*>(s_desc + desc_cap);
  float* const s_kprev = reinterpret_cast<float*>(s_tprev + desc_cap);
  // where each run lies in its row (the index of its first plastic weight is
  // the row's start plus that; BF16 streams count from twice the row's start)
  uint32_t* const s_at = reinterpret_cast<uint32_t*>(s_kprev + desc_cap);
  __shared__ unsigned long long s_pl[2];             // plastic updates, truncations
  __shared__ FixScale s_fx;
  const uint32_t TW = v.tile_w;
  const uint32_t W = (uint32_t)v.window;
  const uint32_t cells = W * TW;
  const bool two = v.acc_words == 2;
  const uint32_t acc_len = two ? 2 * cells : cells;
  const uint32_t tgt_lo = tile * TW;
  const unsigned lane = threadIdx.x & 31u;
  const uint32_t warp = threadIdx.x >> 5;
  SpikeEntry pre[1];
  if (threadIdx.x < desc_cap && threadIdx.x < v.list_cap) pre[0] = list[threadIdx.x];
  ListView lv;
  lv.n_sp = (uint32_t)(*reinterpret_cast<volatile unsigned long long*>(pair_p) >> 32);
  lv.t_now = v.ctl->t_now;
  lv.base = lv.t_now + v.d_min;
  lv.inwin = true;
  const uint32_t n_sp = lv.n_sp;
  const long long base = lv.base;
  if (threadIdx.x == 0) s_fx = fix_scale(v, n_sp, true);
  for (uint32_t x = threadIdx.x; x < acc_len; x += blockDim.x) acc_mem[x] = 0;
  // the post-spike times of this tile's targets (rings) and their post
  // traces at the W horizons (t - d) this interval can ask for
  int32_t* const s_rt = acc_mem + acc_len;                             // [hist][TW]
  uint32_t* const s_rn = reinterpret_cast<uint32_t*>(s_rt + v.sp.hist * TW);
  float* const s_km = reinterpret_cast<float*>(s_rn + TW);             // [W][TW]
  const bool tile_plastic = tgt_lo < v.sp.n_exc;
  uint32_t my_pl = 0, my_trunc = 0;
  // first horizon: (interval start) - d_max
  const long long h_lo = base - v.d_min - v.d_max;
  if (threadIdx.x < 2) s_pl[threadIdx.x] = 0ull;
  if (tile_plastic) {
    for (uint32_t x = threadIdx.x; x < TW; x += blockDim.x)
      s_rn[x] = tgt_lo + x < v.n ? v.sp.ring_n[tgt_lo + x] : 0u;
    for (uint32_t x = threadIdx.x; x < v.sp.hist * TW; x += blockDim.x) {
      const uint32_t q = x / TW, jj = x - q * TW;
      if (tgt_lo + jj < v.n)
        s_rt[x] = v.sp.ring_t[(size_t)q * v.pitch + tgt_lo + jj];
    }
    __syncthreads();
    // post trace of target j at horizon h: the trace right after its
    // latest spike at or before h, decayed to h (0 if it never fired)
    const uint32_t hm = v.sp.hist - 1u;
    for (uint32_t x = threadIdx.x; x < W * TW; x += blockDim.x) {
      const uint32_t hi = x / TW, jj = x - hi * TW;
      const int32_t h = (int32_t)(h_lo + hi);
      const uint32_t n = s_rn[jj];
      const int32_t k_min = n > v.sp.hist ? (int32_t)(n - v.sp.hist) : 0;
      float km = 0.f;
      int32_t k = (int32_t)n - 1;
      for (; k >= k_min; --k) {
        const int32_t tp = s_rt[((uint32_t)k & hm) * TW + jj];
        if (tp <= h) {
          km = v.sp.ring_k[(size_t)((uint32_t)k & hm) * v.pitch + tgt_lo + jj] *
               exp2f(-(float)(h - tp) * v.sp.l2_minus);
          break;
        }
      }
      // every kept spike is after h but older ones were dropped: the
      // trace at h is unknown (-1; an update that needs it is counted
      // with the truncated windows)
      s_km[x] = (k < k_min && n > v.sp.hist) ? -1.f : km;
    }
  }
  FixScale fx{};  // thread 0's s_fx, read after the first barrier
  StdpConst sc;
  sc.c_pot = v.sp.c_pot;
  sc.c_dep = v.sp.c_dep;
  sc.mu = v.sp.mu;
  sc.w_max = v.sp.w_max;
  sc.l2_plus = v.sp.l2_plus;
  sc.l2_minus = v.sp.l2_minus;
  sc.hmask = v.sp.hist - 1u;
  const uint32_t magic = cell_magic(TW);

  // one event of run k_run (spike at step t): the synapse's cell, stored weight,
  // plastic weight (pl: of a plastic run) and the index of the latter
  auto event = [&](uint32_t k_run, const SegDesc& sd, int32_t t, bool pl,
                   uint32_t cell, float w, float wv, uint64_t r) {
    if (pl) w = wv;  // (static synapses of a plastic run: the stored weight)
    const uint32_t ds = cell_step(cell, magic), j = cell - ds * TW;
    if (pl && tgt_lo + j < v.sp.n_exc) {
      const uint32_t d = ds + (uint32_t)v.d_base;
      const float km = s_km[(uint32_t)((long long)t - (long long)d - h_lo) * TW + j];
      const StdpOut o = stdp_weight(w, t, d, s_tprev[k_run], s_kprev[k_run], j,
                                    TW, s_rt, fmaxf(km, 0.f), s_rn[j], sc);
      w = o.w;
      v.sp.wp[r] = w;
      ++my_pl;
      my_trunc += o.trunc | (km < 0.f ? 1u : 0u);
    }
    const uint32_t c = (uint32_t)sd.off + cell;
    if (fx.fixed) {
      int hi, lo;
      fixed_split(w, fx, hi, lo);
      atomicAdd(&acc_mem[c], hi);
      if (two && (LAY == kLayF32 || lo != 0)) atomicAdd(&acc_mem[cells + c], lo);
    } else {
      atomicAdd(reinterpret_cast<float*>(acc_mem) + c, w);
    }
    if (COUNT) {
      const uint32_t sl = c / TW;
      atomicAdd(v.counts + (size_t)((uint32_t)(base + sl) & v.slot_mask) * v.pitch +
                    tgt_lo + (c - sl * TW), 1u);
    }
  };
  // synapse idx of a run: the stream's word (weight and cell), the index of
  // its plastic weight
  struct Syn { uint32_t a, c; };
  auto load_syn = [&](const SegDesc& sd, uint32_t idx) {
    Syn x;
    if constexpr (LAY == kLayF32) {
      x.a = __ldcs(reinterpret_cast<const uint32_t*>(v.dat) + sd.beg + idx);
      x.c = __ldcs(v.cells + sd.beg + idx);
    } else {
      // (taken apart only when it is added: no use before the other loads)
      x.a = __ldcs(reinterpret_cast<const uint32_t*>(v.dat) + sd.beg + idx);
      x.c = 0;
    }
    return x;
  };
  auto syn_cell = [&](const Syn& x) { return LAY == kLayF32 ? x.c : x.a & 0xFFFFu; };
  auto syn_w = [&](const Syn& x) {
    return __uint_as_float(LAY == kLayF32 ? x.a : x.a & 0xFFFF0000u);
  };
  auto check = [&](const SegDesc& sd, uint32_t idx, uint32_t cell) {
#if SNN_CHECK
    const uint64_t ti = sd.tgt + idx;
    return cell_in_bounds(v, cell, v.tgts ? v.tgts[ti]
                                          : reinterpret_cast<const uint32_t*>(v.recs)[ti],
                          tgt_lo);
#else
    return true;
#endif
  };

  uint32_t j0 = 0;
  do {
    const uint32_t nb = min(desc_cap, n_sp - j0);
    describe_runs<LAY, 1, true, kListOwn>(v, lv, list, tile, j0, nb, true, pre, nullptr,
                                  nullptr, s_desc, 0u, s_tprev, s_kprev, s_at);
    __syncthreads();
    fx = s_fx;
    for (uint32_t k0 = warp * U; k0 < nb; k0 += kTileWarps * U) {
      Syn r[U][PER];
      float wv[U][PER];
      uint64_t wi[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t j = k0 + (uint32_t)u;
        const bool ok = j < nb;
        const SegDesc sd = ok ? s_desc[j] : SegDesc{};
        const bool pl = tile_plastic && ok && s_kprev[j] >= 0.f;
        wi[u] = !ok ? 0ull : LAY == kLayF32 ? sd.beg : (sd.beg + s_at[j]) >> 1;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
          const uint32_t idx = lane + 32u * q;
          if (idx < sd.len) {
            r[u][q] = load_syn(sd, idx);
            if (pl) wv[u][q] = __ldcs(v.sp.wp + wi[u] + idx);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t j = k0 + (uint32_t)u;
        if (j >= nb) break;  // (uniform across the warp)
        const SegDesc sd = s_desc[j];
        const bool pl = tile_plastic && s_kprev[j] >= 0.f;
        // (the run's step after base - d_base, from a multiple of TW)
        const int32_t t =
            (int32_t)(base - v.d_base) - 256 +
            (int32_t)cell_step((uint32_t)(sd.off + 256 * (int32_t)TW), magic);
#pragma unroll
        for (int q = 0; q < PER; ++q) {
          const uint32_t idx = lane + 32u * q;
          if (idx < sd.len && check(sd, idx, syn_cell(r[u][q])))
            event(j, sd, t, pl, syn_cell(r[u][q]), syn_w(r[u][q]), wv[u][q],
                  wi[u] + idx);
        }
        for (uint32_t idx = 32u * PER + lane; idx < sd.len; idx += 32u) {
          const Syn x = load_syn(sd, idx);
          const float w = pl ? __ldcs(v.sp.wp + wi[u] + idx) : 0.f;
          if (check(sd, idx, syn_cell(x)))
            event(j, sd, t, pl, syn_cell(x), syn_w(x), w, wi[u] + idx);
        }
      }
    }
    j0 += nb;
    __syncthreads();  // s_desc is rewritten by the next batch
  } while (j0 < n_sp);
  flush_tile<false, false>(v, fx, two, acc_mem, tgt_lo, base);
  // one pair of atomics per warp, one per CTA
  unsigned long long a = my_pl, b = my_trunc;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(kFull, a, o);
    b += __shfl_xor_sync(kFull, b, o);
  }
  if (lane == 0 && (a | b)) {
    atomicAdd(&s_pl[0], a);
    atomicAdd(&s_pl[1], b);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_pl[0] | s_pl[1]) {
      atomicAdd(&v.ctl->plastic_events, s_pl[0]);
      atomicAdd(&v.ctl->stdp_truncated, s_pl[1]);
    }
    finish_list(v, pair_p, done_p, advance_time, false);
  }
}

// A caller's list whose steps span more than the window: known only on the
// device, so called from the other mode's kernel, which has nothing left to do.
template <int LAY, int KIND>
__device__ __forceinline__ void deliver_tile_outside(
    const NetView& v, unsigned long long* pair_p, unsigned int* done_p,
    const SpikeEntry* __restrict__ list, uint32_t tile, int* acc_mem,
    uint32_t desc_off, uint32_t desc_cap) {
  deliver_tile_body<LAY, false, KIND, kAddAny>(v, pair_p, done_p, list, 0, tile,
                                               acc_mem, desc_off, desc_cap);
}

template <int LAY, bool COUNT, int KIND, int MODE>
__global__ void __launch_bounds__(kTileThreads, 1)
k_deliver_tiled(const __grid_constant__ NetView v, unsigned long long* pair_p,
                unsigned int* done_p, const SpikeEntry* __restrict__ list,
                int advance_time, uint32_t desc_off, uint32_t desc_cap) {
  extern __shared__ __align__(16) int acc_mem[];
  deliver_tile_body<LAY, COUNT, KIND, MODE>(v, pair_p, done_p, list, advance_time,
                                            blockIdx.x, acc_mem, desc_off, desc_cap);
  // the next update may be scheduled once every CTA got here
  asm volatile("griddepcontrol.launch_dependents;");
}

// Plastic nets: one tile of plastic targets, or up to tile_grp static tiles
// one after another in the same shared memory.
template <int LAY, bool COUNT>
__global__ void __launch_bounds__(kTileThreads, 1)
k_deliver_plastic(NetView v, unsigned long long* pair_p, unsigned int* done_p,
                  const SpikeEntry* __restrict__ list, int advance_time,
                  uint32_t desc_off, uint32_t desc_cap) {
  extern __shared__ __align__(16) int acc_mem[];
  uint32_t t0 = blockIdx.x, t1 = blockIdx.x + 1u;
  if (blockIdx.x >= v.pl_tiles) {
    t0 = v.pl_tiles + (blockIdx.x - v.pl_tiles) * v.tile_grp;
    t1 = min(t0 + v.tile_grp, v.n_tiles);
  }
  for (uint32_t t = t0; t < t1; ++t) {
    if (t > t0) __syncthreads();  // the previous tile's last reads
    deliver_tile_plastic<LAY, COUNT>(v, pair_p, done_p, list, advance_time, t,
                                     acc_mem, desc_off, desc_cap);
  }
  asm volatile("griddepcontrol.launch_dependents;");
}

// A served net's tile, its pending interval list (advancing the net's clock).
// ANY: some of the launch's nets add their lists element by element (those
// bodies out of line: beside the others they would cost them registers).
template <int LAY, int MODE>
__device__ __forceinline__ void serve_tile_body(const NetView& v, uint32_t tile,
                                                int* acc_mem, uint32_t desc_off,
                                                uint32_t desc_cap) {
  deliver_tile_body<LAY, false, kListOwn, MODE>(
      v, &v.ctl->pair, &v.ctl->done, v.list, 1, tile, acc_mem, desc_off, desc_cap);
}
template <int LAY, int MODE>
__device__ __noinline__ void serve_tile_call(const NetView& v, uint32_t tile,
                                             int* acc_mem, uint32_t desc_off,
                                             uint32_t desc_cap) {
  serve_tile_body<LAY, MODE>(v, tile, acc_mem, desc_off, desc_cap);
}
template <int LAY, bool ANY>
__device__ __forceinline__ void serve_tile_lay(const NetView& v, uint32_t tile,
                                               int* acc_mem, uint32_t desc_off,
                                               uint32_t desc_cap) {
  if constexpr (!ANY)
    serve_tile_body<LAY, kAddVectors>(v, tile, acc_mem, desc_off, desc_cap);
  else if (v.own_mode == kAddVectors)
    serve_tile_call<LAY, kAddVectors>(v, tile, acc_mem, desc_off, desc_cap);
  else
    serve_tile_call<LAY, kAddAny>(v, tile, acc_mem, desc_off, desc_cap);
}
template <int FMT, bool ANY>
__device__ __forceinline__ void serve_tile(const NetView& v, uint32_t tile,
                                           int* acc_mem, uint32_t desc_off,
                                           uint32_t desc_cap) {
  if (v.lay == kLayHom)
    serve_tile_lay<kLayHom, ANY>(v, tile, acc_mem, desc_off, desc_cap);
  else if (FMT == SNN_W_BF16_8B && v.lay == kLayI16)
    serve_tile_lay<kLayI16, ANY>(v, tile, acc_mem, desc_off, desc_cap);
  else
    serve_tile_lay<FMT == SNN_W_FP32_12B ? kLayF32 : kLayJ16, ANY>(
        v, tile, acc_mem, desc_off, desc_cap);
}

// All nets of a batch in one launch: CTA b delivers tile bmap[b].y of net
// bmap[b].x.
template <int FMT, bool ANY>
__global__ void __launch_bounds__(kTileThreads, 1)
k_deliver_tiled_batch(const BatchNet* __restrict__ nets,
                      const uint2* __restrict__ bmap, uint32_t desc_off,
                      uint32_t desc_cap) {
  extern __shared__ __align__(16) int acc_mem[];
  // (the net's view once per CTA in shared memory: a copy per thread goes to
  // local memory)
  __shared__ NetView s_v;
  const uint2 m = bmap[blockIdx.x];
  load_shared(&s_v, &nets[m.x].v);
  __syncthreads();
  serve_tile<FMT, ANY>(s_v, m.y, acc_mem, desc_off, desc_cap);
}

// ---------------------------------------------------------------------------
// Many intervals in one launch.
//
// k_simulate runs the time-driven cycle -- update, exchange of the interval's
// spikes, delivery -- for a whole call of a net with at most a tile per SM: a
// cooperative launch, CTA r owning target tile r with its neurons.  Per
// interval a CTA delivers the previous interval's list into its tile's
// accumulator, updates the tile's neurons straight from it (what later steps
// get goes on to the ring buffer), and publishes its spikes; nothing else
// crosses CTAs.  Each CTA has its own region of the interval's list and a flag
// word {interval, spike count}; the wait for all flags is the exchange's
// barrier, and the counts it reads are the list's lengths: one store and one
// load of latency, no counter shared by all.  Flags and lists alternate
// between two sets: a CTA writes a set again only after every CTA has
// published the interval between, hence has read the set.
//
// The separate kernels spent, per interval of the 112,500-neuron network, 13
// us in the update and 22 us in the delivery, of which 12 us with an empty
// list: launch, list and clock reads, clearing, the ring buffer written by one
// kernel and read and cleared by the next.  Here the state stays in registers,
// the drive is drawn while the list's index words arrive, the rows of the
// neurons that just fired are requested into L2, and all threads of a CTA form
// the steps' inputs however few targets it has.  What bounds it: instructions
// of the accumulation (about 11 of 30 us an interval at 112,500 neurons), then
// latencies in series.  Per interval, two kernels in a graph on whole records,
// on split stores, and here: 1,250 neurons FP32 13.9, 13.6, 8.5 us;
// 20,003 BF16 19.7, 18.2, 13.9; 112,500 FP32 48.0, 34.0, 30.2.  Nets of more
// tiles than SMs keep the two kernels (562,500 neurons: 143 us against 178
// with two tiles a CTA here).
// ---------------------------------------------------------------------------
constexpr uint32_t kSimMaxCtas = 256;
constexpr uint32_t kSimMaxSteps = 32;     // steps of an interval (one spike mask)
constexpr uint32_t kDriveBits = 10;       // leading bits of a draw per table entry

// Cells' kind by layout: the persistent cycle runs only nets whose scales (and
// counts) exist for every interval.
template <int LAY> struct SimCell {
  static constexpr int kKind = LAY == kLayHom ? kCellCounts
                             : LAY == kLayI16 ? kCellOne : kCellTwo;
  static constexpr bool kTwo = LAY == kLayF32 || LAY == kLayJ16;
};

// draw(seed, id, block, 2) with the seed's round keys (seed + r x the Weyl
// increments) as kernel constants.
__device__ __forceinline__ U4 draw_keys(const SimShared& sh, uint32_t id, uint32_t block) {
  U4 c{id, block, 0u, 2u};
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t m0 = (uint64_t)0xD2511F53u * c.x;
    const uint64_t m1 = (uint64_t)0xCD9E8D57u * c.z;
    c = U4{(uint32_t)(m1 >> 32) ^ c.y ^ sh.key[2 * r], (uint32_t)m1,
           (uint32_t)(m0 >> 32) ^ c.w ^ sh.key[2 * r + 1], (uint32_t)m0};
  }
  return c;
}

// Poisson counts of four draws, a byte each.  tab[w >> 22] holds the outcomes below the draw's
// bucket (bits 22 on) plus 2^22 less the one threshold inside it: adding the
// draw's low bits carries exactly when the draw reaches that threshold.
// Buckets with more thresholds (the tail) have bit 31 set and are searched.
__device__ __forceinline__ uint32_t drive_counts(const U4& d, const uint32_t* tab,
                                                 const uint32_t* thr, int n_thr) {
  constexpr int kS = 32 - kDriveBits;
  constexpr uint32_t kLow = (1u << kS) - 1u;
  const uint32_t w[4] = {d.x, d.y, d.z, d.w};
  uint32_t e[4], out = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) e[q] = tab[w[q] >> kS];
#pragma unroll
  for (int q = 0; q < 4; ++q) out |= ((e[q] + (w[q] & kLow)) >> kS) << (8 * q);
  if ((int)(e[0] | e[1] | e[2] | e[3]) < 0) {
    out = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t k = (e[q] + (w[q] & kLow)) >> kS;
      if ((int)e[q] < 0) {
        k = (e[q] & 0x7FFFFFFFu) >> kS;
        while ((int)k < n_thr - 1 && w[q] >= thr[k]) ++k;
      }
      out |= k << (8 * q);
    }
  }
  return out;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long x;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
  return x;
}
__device__ __forceinline__ void st_release_u64(unsigned long long* p, unsigned long long x) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(x) : "memory");
}

// Requests the bytes [p, p + bytes) into L2 (whole 16-byte units around them).
__device__ __forceinline__ void prefetch_l2(const void* p, uint64_t bytes) {
  const uint64_t a = reinterpret_cast<uint64_t>(p) & ~15ull;
  const uint64_t e = (reinterpret_cast<uint64_t>(p) + bytes + 15ull) & ~15ull;
  if (e > a)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                 ::"l"(a), "r"((uint32_t)(e - a)) : "memory");
}
// The stream of the row [beg, end) that a delivery of its source reads.
template <int LAY>
__device__ __forceinline__ void prefetch_stream(const NetView& v, uint64_t beg,
                                                uint64_t len) {
  const char* d = reinterpret_cast<const char*>(v.dat);
  if constexpr (LAY == kLayHom) {
    prefetch_l2(d + 2 * beg * v.row_mul, 2 * len);
  } else {
    prefetch_l2(d + 4 * beg * v.row_mul, 4 * len);
    if constexpr (LAY == kLayF32)
      prefetch_l2(reinterpret_cast<const char*>(v.cells) + 2 * beg, 2 * len);
  }
}

__device__ __forceinline__ uint32_t ld_list(const uint32_t* p) {
  uint32_t x;
  asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
  return x;
}

__device__ __forceinline__ uint64_t ld_row(const uint64_t* p) {
  uint64_t x;
  asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
  return x;
}

// LIMITED: the limit of a wait is the launch's (tests); a parameter compared in the
// poll loop costs 2 % at 20,003 neurons.
template <int LAY, bool LIMITED>
__global__ void __launch_bounds__(kTileThreads, 1)
k_simulate(const __grid_constant__ NetView v, const __grid_constant__ UpdConst c,
           SimShared sh, int n_iv, int n_steps, int last_steps,
           uint32_t drv_off, uint32_t desc_off, uint32_t desc_cap,
           uint32_t pf_rows) {
  extern __shared__ __align__(16) int acc[];
  // drive of the interval to come: [4-step block][target], a byte a step
  uint32_t* const s_drv =
      reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(acc) + drv_off);
  SegDesc* const s_desc =
      reinterpret_cast<SegDesc*>(reinterpret_cast<char*>(acc) + desc_off);
  __shared__ uint32_t s_tab[1u << kDriveBits];
  __shared__ uint32_t s_thr[kMaxPoisson];
  __shared__ uint32_t s_start[kSimMaxCtas + 1];  // list index of each CTA's first
  __shared__ uint32_t s_wsum[kSimMaxCtas / 32];
  __shared__ uint32_t s_cnt;                     // spikes published this interval
  __shared__ int s_bad;
  __shared__ FixScale s_fx;
  __shared__ unsigned long long s_sum[2];
  constexpr int KIND = SimCell<LAY>::kKind;
  constexpr bool TWO = SimCell<LAY>::kTwo;
  const uint32_t G = gridDim.x, r = blockIdx.x;
  const uint32_t tid = threadIdx.x, lane = tid & 31u;
  const uint32_t TW = v.tile_w, W = (uint32_t)v.window, cells = W * TW;
  const uint32_t acc_s = (uint32_t)__cvta_generic_to_shared(acc);
  const uint32_t magic = cell_magic(TW);
  const bool single = TW <= (uint32_t)kTileThreads;  // one neuron a thread
  const uint32_t lo = r * TW, x_end = min(TW, v.n - lo);  // this CTA's targets
  const bool drive = c.n_thr > 0;

  // the drive's table and thresholds, an empty accumulator
  for (uint32_t k = tid; k < (uint32_t)c.n_thr; k += kTileThreads) s_thr[k] = c.thr[k];
  for (uint32_t x = tid; x < (TWO ? 2 * cells : cells); x += kTileThreads) acc[x] = 0;
  if (tid == 0) {
    s_cnt = 0;
    s_bad = 0;
    s_sum[0] = s_sum[1] = 0ull;
    s_fx = FixScale{0, 0, 0, 1.f, 1.f, 1.f, 1.f};
  }
  if (drive) {
    constexpr uint32_t kSpan = 1u << (32 - kDriveBits);
    const uint32_t lo = tid * kSpan;  // (one entry a thread)
    uint32_t k = 0, inside = 0, thr = 0;
    for (int m = 0; m < c.n_thr - 1; ++m) {
      const uint32_t x = c.thr[m];
      if (x <= lo) ++k;
      else if (x - lo < kSpan) { ++inside; thr = x; }
    }
    s_tab[tid] = inside > 1 ? 0x80000000u | (k << (32 - kDriveBits))
                            : (k << (32 - kDriveBits)) + (inside ? kSpan - (thr - lo) : 0u);
  }
  static_assert((1u << kDriveBits) == (uint32_t)kTileThreads, "an entry a thread");
  // (clocks stay below 2^31)
  int t = (int)*reinterpret_cast<volatile long long*>(&v.ctl->t_now);
  unsigned long long logged = *reinterpret_cast<volatile unsigned long long*>(&v.ctl->log_count);
  unsigned long long my_events = 0, my_spikes = 0;
  // (simulate_fits has shown on the host that the scales, and the counts of uniform
  // weights, exist for every list; they do if they do for the largest one's bound,
  // and this says so if the device finds otherwise)
  if (r == 0 && tid == kTileThreads - 1) {
    const FixScale f = fix_scale(v, 0xFFFFFFFFull, true);
    if (!(f.fixed && (LAY != kLayHom || f.packed)))
      atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_SCALES);
  }
  // (a net whose cycle once gave up stays as it is until its errors are cleared:
  // its CTAs had stopped at different steps; a CTA that set out beside one that
  // finds this finds `stop` set)
  if (__syncthreads_or(tid == 0 &&
                       (*reinterpret_cast<volatile unsigned int*>(&v.ctl->error_flags) &
                        (unsigned)SNN_ERRF_TIMEOUT)))
    return;

  // state of this thread's neuron, kept over the launch when it has only one
  float V = 0.f, I = 0.f, J = 0.f;
  int refr = 0;
  if (single && tid < x_end) {
    const uint32_t i = lo + tid;
    V = v.V[i];
    I = v.I[i];
    J = v.J[i];
    refr = v.refr[i];
  }

  const uint32_t* list = nullptr;  // the list published last
  uint32_t n_sp = 0;
  int t_list = 0;                  // its first step
  // one round more than intervals: the last delivers the last list into the
  // ring buffer
  int iv = 0;
  for (; iv <= n_iv; ++iv) {
    const int steps = iv == n_iv ? 0 : iv == n_iv - 1 ? last_steps : n_steps;
    uint32_t* const my_list =
        sh.list + (size_t)((uint32_t)(iv & 1) * G + r) * sh.region;
    // step of the window's slot 0: the round's first step (the interval is the
    // minimum delay), but after a last, shorter interval
    const int tb = iv == n_iv ? t_list + v.d_min : t;
    const int b0 = tb >> 2, a0 = tb & 3;  // the round's first 4-step block
    const uint32_t nb_up = steps ? (uint32_t)((a0 + steps + 3) >> 2) : 0u;
    // draws the drive of the steps to come (while the index words arrive)
    auto draw_drive = [&]() {
      if (!drive) return;
      for (uint32_t k = tid; k < nb_up * TW; k += kTileThreads) {
        const uint32_t j = cell_step(k, magic), x = k - j * TW;
        s_drv[k] = drive_counts(draw_keys(sh, v.g0 + lo + x, (uint32_t)b0 + j),
                                s_tab, s_thr, c.n_thr);
      }
    };
    // (1) the list's events for this tile into the accumulator
    if (iv > 0 && tid == kTileThreads - 1) s_fx = fix_scale(v, n_sp, true);
    uint32_t j0 = 0;
    do {
      const uint32_t nb = min(desc_cap, n_sp - j0);
      for (uint32_t k0 = tid; k0 < nb || k0 == tid; k0 += 2 * kTileThreads) {
        uint32_t e[2] = {0u, 0u}, ra[2] = {0u, 0u}, rb[2] = {0u, 0u};
        uint64_t row[2] = {0ull, 0ull};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (k0 + u * kTileThreads >= nb) continue;
          // the CTA whose region holds list entry g: the last one that
          // starts at or before it (empty ones start where the next does)
          const uint32_t g = j0 + k0 + u * kTileThreads;
          uint32_t at = 0, hi = G;
          while (hi - at > 1) {
            const uint32_t mid = (at + hi) >> 1;
            if (s_start[mid] <= g) at = mid; else hi = mid;
          }
#if SNN_CHECK
          if (!flag_check(v, at < G && g - s_start[at] < sh.region)) {
            e[u] = 0xFFFFFFFFu;
            continue;
          }
#endif
          e[u] = ld_list(list + (size_t)at * sh.region + (g - s_start[at]));
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (k0 + u * kTileThreads >= nb) continue;
          const uint32_t src = e[u] & 0xFFFFFFu;
#if SNN_CHECK
          if (!flag_check(v, src < v.n_src && (int)(e[u] >> 24) < v.d_min)) {
            e[u] = 0u;
            continue;  // (an empty run)
          }
#endif
          const uint32_t* to = v.tile_off + (uint64_t)src * (v.n_tiles + 1) + r;
          ra[u] = ld_list(to);
          rb[u] = ld_list(to + 1);
          row[u] = ld_row(v.row_ptr + src);
        }
        if (j0 == 0 && k0 == tid) draw_drive();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t k = k0 + u * kTileThreads;
          if (k >= nb) continue;
          SegDesc sd;
#if SNN_CHECK
          const uint64_t row_end = v.row_ptr[(e[u] & 0xFFFFFFu) + 1];
          if (!flag_check(v, ra[u] <= rb[u] && (rb[u] == 0 || row[u] + rb[u] <= row_end)))
            rb[u] = ra[u];
          sd.tgt = v.fmt == SNN_W_FP32_12B ? row[u] + ra[u]
                                           : 2 * row[u] + (row_end - row[u]) + ra[u];
#endif
          place_run<LAY>(v, row[u] * v.row_mul + ra[u], rb[u] - ra[u], &sd);
          // (base = t_list + d_min)
          sd.off = ((int32_t)(e[u] >> 24) - v.d_min + v.d_base) * (int32_t)TW;
          if (LAY == kLayHom && (e[u] & 0xFFFFFFu) >= v.hom_split) sd.len |= 0x80000000u;
          s_desc[k] = sd;
        }
      }
      uint32_t lg = (uint32_t)v.lg_cycle;
      while (lg < 5u && (nb << (lg + 1u)) <= (uint32_t)kTileThreads) ++lg;
      __syncthreads();
      if (nb)
        add_runs_call<LAY>(reinterpret_cast<const char*>(v.dat),
                           reinterpret_cast<const char*>(v.cells), s_desc, nb,
                           acc_s, TWO ? 4u * cells : 0u, lg,
                           SplitScale{s_fx.scale_hs, s_fx.scale_s}
                               SNN_CHECKED(RunCheck{&v, lo, cells}));
      j0 += nb;
      if (j0 < n_sp) __syncthreads();  // s_desc is rewritten by the next batch
    } while (j0 < n_sp);
    // (2) the input of every step and target: the ring buffer's value and
    // the list's sum and drive, as a float in the cell's place; later steps'
    // sums go on to the ring buffer.  All threads take part, however few
    // targets the tile has, four cells at a time.
    {
      const FixScale fx = s_fx;
      const CellValue val(v, fx);
      const uint32_t n_in = (uint32_t)steps * TW;
      bool first = true;
      for (uint32_t k0 = tid; first || k0 < n_in; k0 += 4 * kTileThreads) {
        float in[4];
        uint32_t st[4], at[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t k = k0 + q * kTileThreads;
          st[q] = cell_step(k, magic);
          at[q] = k - st[q] * TW;
          in[q] = 0.f;
          if (k < n_in && at[q] < x_end)
            in[q] = __ldcg(v.rb + lo + at[q] +
                           (size_t)((uint32_t)(tb + st[q]) & v.slot_mask) * v.pitch);
        }
        if (first) __syncthreads();  // the sums are complete
        first = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t k = k0 + q * kTileThreads;
          if (k >= n_in || at[q] >= x_end) continue;
          const float a = val.get<KIND>(acc, k, cells);
          if (__float_as_uint(in[q]) != 0u)
            v.rb[lo + at[q] + (size_t)((uint32_t)(tb + st[q]) & v.slot_mask) * v.pitch] = 0.f;
          if (a != 0.f) in[q] += a;
          if (drive) {
            const uint32_t u = (uint32_t)a0 + st[q];
            in[q] += c.w_ext * (float)((s_drv[(u >> 2) * TW + at[q]] >> (8u * (u & 3u))) & 0xFFu);
          }
          reinterpret_cast<float*>(acc)[k] = in[q];
          if (TWO) acc[cells + k] = 0;
        }
      }
      if (iv > 0)
        for (uint32_t k = n_in + tid; k < cells; k += kTileThreads) {
          const float a = val.get<KIND>(acc, k, cells);
          if (a != 0.f) {
            const uint32_t sl = cell_step(k, magic);
            red_add_f32(v.rb + lo + (k - sl * TW) +
                            (size_t)((uint32_t)(tb + sl) & v.slot_mask) * v.pitch, a);
          }
          acc[k] = 0;
          if (TWO) acc[cells + k] = 0;
        }
    }
    if (steps == 0) break;
    __syncthreads();
    // (3) the neurons, a thread each, through the interval's steps
    for (uint32_t x0 = 0; x0 < TW; x0 += kTileThreads) {
      const uint32_t x = x0 + tid, i = lo + x;
      const bool live = x < x_end;
      uint32_t mask = 0;
      if (live) {
        if (!single) {
          V = v.V[i];
          I = v.I[i];
          J = v.J[i];
          refr = v.refr[i];
        }
        int* p = acc + x;
        float in = __int_as_float(*p);
        for (int s = 0; s < steps; ++s, p += TW) {
          const float next = s + 1 < steps ? __int_as_float(p[TW]) : 0.f;
          *p = 0;
          if (update_step(c, V, I, J, refr, in)) mask |= 1u << s;
          in = next;
        }
        if (!single) {
          v.V[i] = V;
          v.I[i] = I;
          v.J[i] = J;
          v.refr[i] = refr;
        }
      }
      // this tile's spikes into the CTA's region of the list
      const uint32_t cnt = __popc(mask);
      uint32_t at = 0;
      if (__ballot_sync(kFull, cnt != 0)) {
        uint32_t inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(kFull, inc, o);
          if (lane >= (unsigned)o) inc += y;
        }
        if (lane == 31u) at = atomicAdd(&s_cnt, inc);
        at = __shfl_sync(kFull, at, 31) + inc - cnt;
        uint32_t to = at;
        for (uint32_t m = mask; m; m &= m - 1u, ++to)
          if (to < sh.region)  // (always: simulate_fits)
            my_list[to] = (v.g0 + i) | ((uint32_t)(__ffs(m) - 1) << 24);
      }
      if (x0 + kTileThreads >= TW) {
        // publish: every thread's entries, then the count (the release
        // covers what the barrier ordered before it)
        __syncthreads();
        if (tid == 0)
          st_release_u64(&sh.flags[(uint32_t)(iv & 1) * kSimMaxCtas + r],
                         ((unsigned long long)(iv + 1) << 32) | s_cnt);
      }
      if (cnt) {
        // the deliveries that follow read this source's row of the tile
        // index and, for as many rows as L2 takes, its synapses
        prefetch_row_l2(v, v.g0 + i);
        const uint64_t beg = v.row_ptr[v.g0 + i];
        const uint64_t len = v.row_ptr[v.g0 + i + 1] - beg;
        if (at < pf_rows) prefetch_stream<LAY>(v, beg, len);
        my_events += cnt * len;
        my_spikes += cnt;
        if (v.isi_spikes) {
          int32_t last = v.isi_last[i];
          uint32_t n_isi = v.isi_n[i];
          double s1 = v.isi_sum[i], s2 = v.isi_sq[i];
          for (uint32_t m = mask; m; m &= m - 1u) {
            const int32_t ts = t + __ffs(m) - 1;
            if (last != kNoSpike) {
              const double d = (double)(ts - last);  // exact in FP64
              s1 += d;
              s2 += d * d;
              n_isi += 1u;
            }
            last = ts;
          }
          v.isi_last[i] = last;
          v.isi_spikes[i] += cnt;
          v.isi_n[i] = n_isi;
          v.isi_sum[i] = s1;
          v.isi_sq[i] = s2;
        }
      }
    }
    t_list = t;
    t += steps;
    // (4) every CTA's count (thread k: CTA k's), and where its entries start
    if (tid < kSimMaxCtas) {
      uint32_t n_r = 0;
      if (tid < G) {
        const unsigned long long* f = &sh.flags[(uint32_t)(iv & 1) * kSimMaxCtas + tid];
        unsigned long long x;
        uint32_t polls = 0;
        while ((uint32_t)((x = ld_acquire_u64(f)) >> 32) != (uint32_t)(iv + 1)) {
          ++polls;
          if (polls > (LIMITED ? sh.polls : kSimPolls) ||
              ((polls & 1023u) == 0u &&
               *reinterpret_cast<volatile unsigned int*>(sh.stop))) {
            s_bad = 1;
            break;
          }
        }
        n_r = (uint32_t)x;
      }
      uint32_t inc = n_r;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, o);
        if (lane >= (unsigned)o) inc += y;
      }
      if (lane == 31u) s_wsum[tid >> 5] = inc;
      s_start[tid] = inc - n_r;
    }
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    if (s_bad) break;  // (uniform: read after the barrier)
    n_sp = 0;
    uint32_t before = 0;
#pragma unroll
    for (uint32_t w = 0; w < kSimMaxCtas / 32; ++w) {
      if (w == (tid >> 5)) before = n_sp;
      n_sp += s_wsum[w];
    }
    if (tid < kSimMaxCtas) s_start[tid] += before;
    __syncthreads();
    list = sh.list + (size_t)((uint32_t)(iv & 1) * G) * sh.region;
    // this CTA's spikes into the log, at their place in the list
    if (v.log_cap && tid >= kTileThreads / 2) {
      const uint32_t mine = (r + 1 < G ? s_start[r + 1] : n_sp) - s_start[r];
      for (uint32_t k = kTileThreads - 1 - tid; k < mine; k += kTileThreads / 2) {
        const uint32_t e = ld_list(my_list + k);
        const unsigned long long at = logged + s_start[r] + k;
        if (at < v.log_cap) {
          v.log_src[at] = e & 0xFFFFFFu;
          v.log_t[at] = t_list + (int32_t)(e >> 24);
        } else {
          atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_SPIKE_LOG);
        }
      }
    }
    logged += n_sp;
  }
  if (s_bad && tid == 0) {
    // a wait ran out: the others leave as well
    atomicExch(sh.stop, 1u);
    atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_TIMEOUT);
  }
  // (a launch that gives up leaves state, ring buffer, log and clock unusable)
  if (single && tid < x_end) {
    const uint32_t i = lo + tid;
    v.V[i] = V;
    v.I[i] = I;
    v.J[i] = J;
    v.refr[i] = refr;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    my_events += __shfl_xor_sync(kFull, my_events, o);
    my_spikes += __shfl_xor_sync(kFull, my_spikes, o);
  }
  if (lane == 0 && my_spikes) {
    atomicAdd(&s_sum[0], my_events);
    atomicAdd(&s_sum[1], my_spikes);
  }
  __syncthreads();
  if (tid == 0) {
    if (s_sum[1]) {
      atomicAdd(&v.ctl->events, s_sum[0]);
      atomicAdd(&v.ctl->spikes, s_sum[1]);
    }
    // the last CTA to end commits the clock and the log's length, if every CTA
    // got through all intervals (all read both before this)
    __threadfence();
    if (atomicAdd(sh.done, 1u) == G - 1 &&
        *reinterpret_cast<volatile unsigned int*>(sh.stop) == 0u) {
      v.ctl->t_now = t;
      v.ctl->iv_steps = last_steps;
      if (v.log_cap) v.ctl->log_count = logged;
    }
  }
}

// ---------------------------------------------------------------------------
// Persistent serving kernel: one launch advances every admitted net by its
// own number of intervals.  Each net is a chain of items -- per interval its
// update blocks, then its delivery tiles -- with the dependencies of the
// time-driven cycle (Section 2.1): an interval's delivery reads the spike
// list its update wrote, and the next update reads the ring buffer that
// delivery filled.  A CTA claims the first ready item of the first net
// (nets are ordered by size, smallest first) and runs it; so small nets
// keep advancing while large ones take the remaining CTAs, and no net waits
// for the pace of another.  Deadlock-free: an item is claimed only when its
// dependencies have completed, and no item waits inside.  The only wait is
// a CTA polling for a ready item; it gives up after spin_limit polls
// (ServeCtl.error = SNN_ERRF_TIMEOUT), and every CTA then leaves.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned x;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
  return x;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// The two kinds of item, compiled out of line (each keeps its own register
// allocation instead of sharing one with the other and the claim loop).
__device__ __noinline__ void serve_update(const NetView& v, const UpdConst& c,
                                          int n_steps, uint32_t block) {
  update_body<false, true>(v, c, n_steps, 1, 0, block);
}
template <int FMT, bool ANY>
__device__ __noinline__ void serve_deliver(const NetView& v, uint32_t tile,
                                           int* acc_mem, uint32_t desc_off,
                                           uint32_t desc_cap) {
  serve_tile<FMT, ANY>(v, tile, acc_mem, desc_off, desc_cap);
}

template <int FMT, bool ANY>
__global__ void __launch_bounds__(kTileThreads, 1)
k_serve(const BatchNet* __restrict__ nets, ServeNet* sn, ServeCtl* ctl,
        uint32_t n_nets, uint32_t desc_off, uint32_t desc_cap,
        unsigned long long spin_limit) {
  extern __shared__ __align__(16) int acc_mem[];
  __shared__ UpdConst s_c;
  __shared__ int s_state;      // 0: run s_net/s_item, 1: all claimed, 2: error
  __shared__ uint32_t s_net, s_item;
  for (;;) {
    if (threadIdx.x == 0) {
      int st = 1;
      unsigned long long polls = 0;
      unsigned nap = 32;  // ns between polls, doubling up to 256 while idle
      for (;;) {
        if (*reinterpret_cast<volatile unsigned*>(&ctl->error)) {
          st = 2;
          break;
        }
        bool left = false, got = false;
        for (uint32_t j = 0; j < n_nets && !got; ++j) {
          volatile ServeNet& q = sn[j];
          const unsigned per = q.ub + q.nt, n_items = q.n_items;
          for (;;) {
            const unsigned k = q.next;
            if (k >= n_items) break;
            left = true;
            const unsigned r = k / per, w = k - r * per;
            const bool ready = w < q.ub ? q.del_done >= r * q.nt
                                        : q.upd_done >= (r + 1) * q.ub;
            if (!ready) break;
            if (atomicCAS(&sn[j].next, k, k + 1) == k) {
              if (k == 0) sn[j].t_first = global_ns();
              s_net = j;
              s_item = k;
              got = true;
              break;
            }
          }
        }
        if (got) {
          st = 0;
          break;
        }
        if (!left) break;  // every item of every net is claimed
        if (++polls > spin_limit) {
          atomicOr(&ctl->error, (unsigned)SNN_ERRF_TIMEOUT);
          st = 2;
          break;
        }
        __nanosleep(nap);
        nap = nap < 256 ? 2 * nap : 256;
      }
      s_state = st;
    }
    __syncthreads();
    if (s_state != 0) break;
    const uint32_t j = s_net, k = s_item;
    ServeNet& q = sn[j];
    const unsigned per = q.ub + q.nt, r = k / per, w = k - r * per;
    const bool upd = w < q.ub;
    // every thread acquires what the item depends on (its writers released
    // it with a fence before counting their item done)
    ld_acquire_u32(upd ? &q.del_done : &q.upd_done);
    const NetView& v = nets[j].v;
    if (upd) {
      const uint32_t* src = reinterpret_cast<const uint32_t*>(&nets[j].c);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&s_c);
      for (uint32_t x = threadIdx.x; x < sizeof(UpdConst) / 4; x += blockDim.x)
        dst[x] = src[x];
      __syncthreads();
      serve_update(v, s_c, nets[j].n_steps, w);
    } else {
      serve_deliver<FMT, ANY>(v, w - q.ub, acc_mem, desc_off, desc_cap);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      atomicAdd(upd ? &q.upd_done : &q.del_done, 1u);
      atomicMax(&q.t_last, global_ns());
    }
  }
}

// ---------------------------------------------------------------------------
// Caller's spike list -> entries with chunk prefix sums (one CTA).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024)
k_prepare_external(NetView v, const uint32_t* __restrict__ src,
                   const int32_t* __restrict__ tt, uint32_t n,
                   SpikeEntry* out, unsigned long long* pair_p) {
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_carry;
  __shared__ int s_tmin, s_tmax;
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_carry = 0;
    s_tmin = 0x7FFFFFFF;
    s_tmax = -0x7FFFFFFF - 1;
  }
  unsigned long long deg_sum = 0;
  int tmin = 0x7FFFFFFF, tmax = -0x7FFFFFFF - 1;
  bool bad = false;
  __syncthreads();
  for (uint32_t base = 0; base < n; base += blockDim.x) {
    const uint32_t i = base + threadIdx.x;
    uint32_t s = 0xFFFFFFFFu, nch = 0;
    int32_t t = 0;
    if (i < n) {
      s = src[i];
      t = tt[i];
      tmin = min(tmin, t);
      tmax = max(tmax, t);
      if (s < v.n_src) {
        uint64_t b = v.row_ptr[s], e = v.row_ptr[s + 1];
        nch = row_chunks(b, e, v.chunk);
        deg_sum += e - b;
      } else {
        s = 0xFFFFFFFFu;
        bad = true;
      }
    }
    uint32_t incl = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= (unsigned)o) incl += y;
    }
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      uint32_t x = lane < (blockDim.x >> 5) ? s_warp[lane] : 0u;
      uint32_t xi = x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(kFull, xi, o);
        if (lane >= (unsigned)o) xi += y;
      }
      s_warp[lane] = xi - x;  // exclusive over warps
    }
    __syncthreads();
    const uint32_t carry = s_carry;
    if (i < n) {
      SpikeEntry en;
      en.src = s;
      en.t = t;
      en.choff = carry + s_warp[wid] + incl - nch;
      en.pad = 0;
      out[i] = en;
    }
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) s_carry = carry + s_warp[wid] + incl;
    __syncthreads();
  }
  // block reduction of deg_sum
  for (int o = 16; o > 0; o >>= 1) deg_sum += __shfl_xor_sync(kFull, deg_sum, o);
  if (lane == 0 && deg_sum) atomicAdd(&v.ctl->events, deg_sum);
  atomicMin(&s_tmin, tmin);
  atomicMax(&s_tmax, tmax);
  if (__syncthreads_or(bad) && threadIdx.x == 0)
    atomicOr(&v.ctl->error_flags, (unsigned)SNN_ERRF_BAD_SOURCE);
  if (threadIdx.x == 0) {
    *pair_p = ((unsigned long long)n << 32) | (unsigned long long)s_carry;
    v.ctl->ext_tmin = s_tmin;
    v.ctl->ext_tmax = s_tmax;
  }
}

// grid of the atomic delivery (SMs x resident blocks), computed on first use
std::atomic<int> g_deliver_blocks[2];

template <int FMT>
int deliver_blocks_for() {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_deliver<FMT, false>,
                                                kDelThreads, 0);
  if (per < 1) per = 1;
  return sms * per;
}

}  // namespace

// q - s of the kernel's fix_scale for event bound e and max|w| (-1: FP32),
// computed on the host with the same steps.
int fixed_qs_host(uint64_t e, double max_abs_w) {
  const float mw = (float)max_abs_w;
  if (e == 0 || e >= (1ull << 30) || !(mw > 0.f) || !(mw <= 3.0e38f)) return -1;
  const double A = 2147483647.0 - (double)e;
  const double B = (double)e * (double)mw;
  int qs = ilogb(A) - ilogb(B);
  if (B * ldexp(1.0, qs) > A) --qs;
  uint32_t wb;
  memcpy(&wb, &mw, 4);
  const int wexp = (int)((wb >> 23) & 0xFFu) - 127 + ((wb & 0x7FFFFFu) ? 1 : 0);
  qs = std::min(qs, 21 - wexp);
  if (qs < 0) return -1;
  return std::min(qs, 100);
}

int add_mode(const NetView& v, uint64_t events) {
  if (v.lay == kLayHom && (events <= 0xFFFFull || v.acc_words == 2))
    return events <= 0xFFFFull ? kAddVectors : kAddWide;
  const int qs = v.lay == kLayRecords ? -1 : fixed_qs_host(events, v.max_abs_w);
  if (qs < 0 || (v.acc_words == 1 && qs < v.acc_qs_min)) return kAddAny;
  return v.lay == kLayHom ? kAddWeighted : kAddVectors;
}
// (the largest bound decides: scales only grow as it shrinks)
int own_add_mode(const NetView& v) {
  return add_mode(v, cell_events(v, ~0u, true));
}

int deliver_grid_size(int fmt) {
  const int k = fmt == SNN_W_FP32_12B ? 0 : 1;
  int b = g_deliver_blocks[k].load(std::memory_order_relaxed);
  if (b == 0) {
    b = fmt == SNN_W_FP32_12B ? deliver_blocks_for<SNN_W_FP32_12B>()
                              : deliver_blocks_for<SNN_W_BF16_8B>();
    g_deliver_blocks[k].store(b, std::memory_order_relaxed);
  }
  return b;
}

cudaError_t launch_init_v(const NetView& v, const UpdConst* c, int random,
                          cudaStream_t s) {
  if (v.n == 0) return cudaSuccess;
  unsigned blocks = (v.n + 255) / 256;
  k_init_state<<<blocks, 256, 0, s>>>(v, c->v_reset, c->v_th - c->v_reset,
                                      c->seed, random);
  return cudaGetLastError();
}

cudaError_t launch_update(const NetView& v, const UpdConst& c, int n_steps,
                          int from_ctl_time, long long t0, cudaStream_t s) {
  unsigned blocks = (v.n + kUpdThreads - 1) / kUpdThreads;
  if (blocks == 0) blocks = 1;
  static std::atomic<int> sms{0};
  if (sms.load(std::memory_order_relaxed) == 0) {
    int dev = 0, m = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
      sms.store(m, std::memory_order_relaxed);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kUpdThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (blocks > 3u * (unsigned)std::max(sms.load(std::memory_order_relaxed), 1))
    return cudaLaunchKernelEx(&cfg, k_update<4>, v, c, n_steps, from_ctl_time, t0);
  return cudaLaunchKernelEx(&cfg, k_update<3>, v, c, n_steps, from_ctl_time, t0);
}

cudaError_t launch_deliver(const NetView& v, unsigned long long* pair,
                           unsigned int* done, const SpikeEntry* list,
                           int advance_time, cudaStream_t s) {
  int blocks = deliver_grid_size(v.fmt);
  if (v.fmt == SNN_W_FP32_12B) {
    if (v.counts)
      k_deliver<SNN_W_FP32_12B, true>
          <<<blocks, kDelThreads, 0, s>>>(v, pair, done, list, advance_time);
    else
      k_deliver<SNN_W_FP32_12B, false>
          <<<blocks, kDelThreads, 0, s>>>(v, pair, done, list, advance_time);
  } else {
    if (v.counts)
      k_deliver<SNN_W_BF16_8B, true>
          <<<blocks, kDelThreads, 0, s>>>(v, pair, done, list, advance_time);
    else
      k_deliver<SNN_W_BF16_8B, false>
          <<<blocks, kDelThreads, 0, s>>>(v, pair, done, list, advance_time);
  }
  return cudaGetLastError();
}

size_t tiled_smem_bytes(const NetView& v) {
  // accumulator; plastic nets: spike-time rings, counts, post-trace table
  return (size_t)v.tile_w *
         ((size_t)v.acc_words * v.window * sizeof(int) +
          (v.plastic ? (size_t)v.sp.hist * 4 + 4 + (size_t)v.window * 4 : 0));
}

// Raise a tiled-delivery kernel's dynamic shared-memory limit to all that
// its static shared memory leaves, once per device (the attribute belongs to
// the kernel on the current device); returns that limit.  `lim` holds one
// entry per device and is safe to fill from several threads.
template <class Kernel>
cudaError_t allow_tile_smem(Kernel kernel, std::atomic<uint32_t>* lim,
                            size_t* dyn_max) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::atomic<uint32_t>& slot = lim[dev & 63];
  const uint32_t have = slot.load(std::memory_order_acquire);
  if (have) {
    *dyn_max = have;
    return cudaSuccess;
  }
  int optin = 0;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  const int dyn = optin - (int)fa.sharedSizeBytes;
  if (dyn <= 0) return cudaErrorInvalidConfiguration;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
  if (e != cudaSuccess) return e;
  slot.store((uint32_t)dyn, std::memory_order_release);
  *dyn_max = (size_t)dyn;
  return cudaSuccess;
}

// Run descriptors go after the accumulator (and the plastic state): at least
// kDescBytes of them (if they fit), and what is left of the shared-memory
// carve-out that this needs anyway -- a larger carve-out would take L1
// capacity, in which the record loads wait, from the kernel: at 562,500
// neurons 32 KB took 7.28 ms a pass (three batches of 2,048 runs), 48 KB of the
// same carve-out 7.07, 72 KB 8.40.
constexpr size_t kDescBytes = 32 * 1024;
struct DescLayout {
  uint32_t off, cap;
  size_t smem;
};
cudaError_t desc_layout(size_t used, size_t dyn_max, bool plastic,
                        DescLayout* out) {
  // (a plastic run also has its source's last spike and its place in the row)
  const size_t per = sizeof(SegDesc) + (plastic ? 12u : 0u);
  const size_t off = (used + 15u) & ~(size_t)15u;
  if (dyn_max < off + 32u * per) return cudaErrorInvalidConfiguration;
  // carve-outs of an SM; a CTA also takes 1 KB and its static memory
  constexpr size_t kCarve[] = {16, 32, 64, 100, 132, 164, 196, 228};
  constexpr size_t kOptin = 227 * 1024;
  const size_t fixed = 1024 + (kOptin > dyn_max ? kOptin - dyn_max : 0);
  size_t room = std::min(kDescBytes, dyn_max - off);
  for (size_t c : kCarve)
    if (c * 1024 >= fixed + off + room) {
      room = std::min(c * 1024 - fixed, dyn_max) - off;
      break;
    }
  const size_t cap = room / per & ~(size_t)1;
  out->off = (uint32_t)off;
  out->cap = (uint32_t)cap;
  out->smem = off + cap * per;
  return cudaSuccess;
}

template <int LAY, bool COUNT, int KIND, int MODE>
cudaError_t launch_tiled_t(const NetView& v, unsigned long long* pair,
                           unsigned int* done, const SpikeEntry* list,
                           int advance_time, cudaStream_t s) {
  static std::atomic<uint32_t> lim[64];
  size_t dm = 0;
  cudaError_t e = allow_tile_smem(k_deliver_tiled<LAY, COUNT, KIND, MODE>, lim, &dm);
  if (e != cudaSuccess) return e;
  DescLayout dl;
  e = desc_layout(tiled_smem_bytes(v), dm, false, &dl);
  if (e != cudaSuccess) return e;
  k_deliver_tiled<LAY, COUNT, KIND, MODE><<<v.n_tiles, kTileThreads, dl.smem, s>>>(
      v, pair, done, list, advance_time, dl.off, dl.cap);
  return cudaGetLastError();
}
template <int LAY, int KIND>
cudaError_t launch_tiled_k(const NetView& v, unsigned long long* pair,
                           unsigned int* done, const SpikeEntry* list, int mode,
                           int advance_time, cudaStream_t s) {
  if (v.counts)
    return launch_tiled_t<LAY, true, KIND, kAddAny>(v, pair, done, list, advance_time, s);
  if (mode == kAddVectors)
    return launch_tiled_t<LAY, false, KIND, kAddVectors>(v, pair, done, list,
                                                         advance_time, s);
  if constexpr (LAY == kLayHom) {
    if (mode == kAddWide)
      return launch_tiled_t<LAY, false, KIND, kAddWide>(v, pair, done, list,
                                                        advance_time, s);
    if (mode == kAddWeighted)
      return launch_tiled_t<LAY, false, KIND, kAddWeighted>(v, pair, done, list,
                                                            advance_time, s);
  }
  return launch_tiled_t<LAY, false, KIND, kAddAny>(v, pair, done, list, advance_time, s);
}

template <int LAY, bool COUNT>
cudaError_t launch_plastic_t(const NetView& v, unsigned long long* pair,
                             unsigned int* done, const SpikeEntry* list,
                             int advance_time, cudaStream_t s) {
  static std::atomic<uint32_t> lim[64];
  size_t dm = 0;
  cudaError_t e = allow_tile_smem(k_deliver_plastic<LAY, COUNT>, lim, &dm);
  if (e != cudaSuccess) return e;
  DescLayout dl;
  e = desc_layout(tiled_smem_bytes(v), dm, true, &dl);
  if (e != cudaSuccess) return e;
  // a CTA per plastic tile, then one per tile_grp static ones
  const uint32_t ctas =
      v.pl_tiles + (v.n_tiles - v.pl_tiles + v.tile_grp - 1u) / v.tile_grp;
  k_deliver_plastic<LAY, COUNT><<<ctas, kTileThreads, dl.smem, s>>>(
      v, pair, done, list, advance_time, dl.off, dl.cap);
  return cudaGetLastError();
}

cudaError_t launch_deliver_tiled(const NetView& v, unsigned long long* pair,
                                 unsigned int* done, const SpikeEntry* list,
                                 uint32_t n_prepared, int advance_time,
                                 cudaStream_t s) {
  if ((v.gx || v.ext_src) && n_prepared) return cudaErrorInvalidValue;
  if (v.plastic) {
    if (v.gx || v.ext_src || n_prepared) return cudaErrorNotSupported;
    if (v.lay == kLayF32)
      return v.counts ? launch_plastic_t<kLayF32, true>(v, pair, done, list, advance_time, s)
                      : launch_plastic_t<kLayF32, false>(v, pair, done, list, advance_time, s);
    return v.counts ? launch_plastic_t<kLayJ16, true>(v, pair, done, list, advance_time, s)
                    : launch_plastic_t<kLayJ16, false>(v, pair, done, list, advance_time, s);
  }
  const uint32_t n_caller = v.ext_src ? v.ext_n : n_prepared;
  const int mode = n_caller ? add_mode(v, cell_events(v, n_caller, false)) : v.own_mode;
#define SNN_TILED(L)                                                            \
  (v.gx ? launch_tiled_k<L, kListGathered>(v, pair, done, list, mode,           \
                                           advance_time, s)                     \
   : v.ext_src ? launch_tiled_k<L, kListRaw>(v, pair, done, list, mode, 0, s) \
   : n_prepared ? launch_tiled_k<L, kListRange>(v, pair, done, list, mode, 0, s) \
                : launch_tiled_k<L, kListOwn>(v, pair, done, list, mode,        \
                                              advance_time, s))
  switch (v.lay) {
    case kLayHom: return SNN_TILED(kLayHom);
    case kLayF32: return SNN_TILED(kLayF32);
    case kLayI16: return SNN_TILED(kLayI16);
    default: return SNN_TILED(kLayJ16);
  }
#undef SNN_TILED
}

bool deliver_raw_fits(const NetView& v, uint32_t n) {
  return v.lay != kLayRecords && n <= kRawMax;
}

cudaError_t launch_deliver_raw(const NetView& v, const uint32_t* src,
                               const int32_t* t, uint32_t n, cudaStream_t s) {
  NetView x = v;
  x.ext_src = src;
  x.ext_t = t;
  x.ext_n = n;
  return launch_deliver_tiled(x, nullptr, nullptr, nullptr, 0u, 0, s);
}

template <int LAY, bool LIMITED>
cudaError_t launch_simulate_t(const NetView& v, const UpdConst& c,
                              const SimShared& sh, uint32_t ctas, int n_iv,
                              int steps, int last_steps, cudaStream_t s) {
  static std::atomic<uint32_t> lim[64];
  size_t dm = 0;
  cudaError_t e = allow_tile_smem(k_simulate<LAY, LIMITED>, lim, &dm);
  if (e != cudaSuccess) return e;
  DescLayout dl;  // after the accumulator and the drive (5 or 9 blocks)
  const size_t drv = ((size_t)v.tile_w * v.window * (SimCell<LAY>::kTwo ? 8u : 4u) + 15u) & ~(size_t)15u;
  const size_t blocks = ((size_t)steps + 6) / 4;
  e = desc_layout(drv + blocks * v.tile_w * 4u, dm, false, &dl);
  if (e != cudaSuccess) return e;
  // as many rows of a CTA's spikes are requested ahead as a third of L2 holds
  // of all CTAs'
  const double row = v.n_src ? (double)v.mean_row * (LAY == kLayHom ? 2.0 : LAY == kLayF32 ? 6.0 : 4.0) : 1.0;
  const uint32_t pf = (uint32_t)std::max(1.0, 40e6 / (std::max(row, 64.0) * ctas));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kTileThreads);
  cfg.dynamicSmemBytes = dl.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // every CTA waits for the others
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, k_simulate<LAY, LIMITED>, v, c, sh, n_iv, steps,
                         last_steps, (uint32_t)drv, dl.off, dl.cap, pf);
  if (e != cudaSuccess) return e;
  // The flags of the launch to come are cleared after this one, not before it:
  // the memset waits for the kernel to end with its writes visible, so a
  // k_update that comes next on the stream, and reads state before its
  // griddepcontrol.wait, can only overlap the memset.
  return cudaMemsetAsync(sh.flags, 0, kSimFlagBytes, s);
}

static int sim_sms() {
  static std::atomic<int> sms[64];
  int dev = 0, m = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  m = sms[dev].load(std::memory_order_relaxed);
  if (m == 0) {
    int coop = 0;
    if (cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        !coop)
      m = -1;
    sms[dev].store(m, std::memory_order_relaxed);
  }
  return m;
}

// Whether the intervals of a net can run in k_simulate: a split store whose
// scales (and counts) exist for every interval, nothing that only the
// separate kernels do (plasticity, counted cells, exchange
// buffers), and lists that fit the interval list's memory.
bool simulate_fits(const NetView& v, const UpdConst& c, int interval,
                   SimShared* sh, uint32_t* ctas) {
  // (a reset at or above the threshold fires at every step, refractory or not)
  if (!(c.v_reset < c.v_th)) return false;
  if (v.lay == kLayRecords || v.plastic || v.counts || v.xbuf ||
      interval < 1 || interval > (int)kSimMaxSteps || v.n_tiles == 0)
    return false;
  const uint64_t e = (uint64_t)v.k_in_max * std::max(v.spikes_per_iv, 1u);
  const int qs = fixed_qs_host(e, v.max_abs_w);
  if (qs < 0 || (v.acc_words == 1 && qs < v.acc_qs_min)) return false;
  // (a list's window starts where the next interval does; room for the drive
  // and some run descriptors beside the accumulator)
  if (interval != v.d_min) return false;
  const uint32_t words = v.lay == kLayF32 || v.lay == kLayJ16 ? 2u : 1u;
  if ((size_t)v.tile_w * (4u * words * v.window + 4u * ((interval + 6) / 4)) >
      (size_t)(210 * 1024))
    return false;
  // (cells and draws are numbered within 16 bits)
  if ((uint64_t)v.tile_w * std::max<uint32_t>(v.window, (interval + 6) / 4) > 0xFFFFull)
    return false;
  if (v.lay == kLayHom && e > 0xFFFFull) return false;
  if (v.lay == kLayJ16 && v.acc_words == 1) return false;
  const int sms = sim_sms();
  // (nets of more tiles than SMs: the separate kernels, whose grids balance
  // their tiles, are faster: 7.15 against 8.90 ms at 562,500 neurons)
  if (sms < 1 || v.n_tiles > std::min<uint32_t>((uint32_t)sms, kSimMaxCtas)) return false;
  const uint32_t G = v.n_tiles;
  const uint64_t region = (uint64_t)v.tile_w * std::max(v.spikes_per_iv, 1u);
  if (2 * G * region * sizeof(uint32_t) > v.list_cap * sizeof(SpikeEntry)) return false;
  sh->list = reinterpret_cast<uint32_t*>(v.list);
  sh->region = (uint32_t)region;
  *ctas = G;
  return true;
}

cudaError_t launch_simulate(const NetView& v, const UpdConst& c,
                            const SimShared& sh, uint32_t ctas, int n_iv,
                            int steps, int last_steps, cudaStream_t s) {
#define SNN_SIMULATE(L)                                                              \
  (sh.polls == kSimPolls                                                             \
       ? launch_simulate_t<L, false>(v, c, sh, ctas, n_iv, steps, last_steps, s)     \
       : launch_simulate_t<L, true>(v, c, sh, ctas, n_iv, steps, last_steps, s))
  switch (v.lay) {
    case kLayHom: return SNN_SIMULATE(kLayHom);
    case kLayF32: return SNN_SIMULATE(kLayF32);
    case kLayI16: return SNN_SIMULATE(kLayI16);
    default: return SNN_SIMULATE(kLayJ16);
  }
#undef SNN_SIMULATE
}

cudaError_t launch_fill_i32(int32_t* p, int32_t value, uint64_t n,
                            cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t blocks = std::min<uint64_t>((n + 255) / 256, 4096);
  k_fill_i32<<<(unsigned)blocks, 256, 0, s>>>(p, value, n);
  return cudaGetLastError();
}

cudaError_t launch_list_to_arrays(const SpikeEntry* list, uint64_t n,
                                  uint32_t* src, int32_t* t, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t blocks = std::min<uint64_t>((n + 255) / 256, 4096);
  k_list_to_arrays<<<(unsigned)blocks, 256, 0, s>>>(list, n, src, t);
  return cudaGetLastError();
}

cudaError_t launch_update_batch(const BatchNet* nets, const uint2* bmap,
                                uint32_t n_blocks, cudaStream_t s) {
  if (n_blocks == 0) return cudaSuccess;
  k_update_batch<<<n_blocks, kUpdThreads, 0, s>>>(nets, bmap);
  return cudaGetLastError();
}

template <int FMT, bool ANY>
static cudaError_t launch_batch_t(const BatchNet* nets, const uint2* bmap,
                                  uint32_t n_ctas, size_t smem, cudaStream_t s) {
  static std::atomic<uint32_t> lim[64];
  size_t dm = 0;
  cudaError_t e = allow_tile_smem(k_deliver_tiled_batch<FMT, ANY>, lim, &dm);
  if (e != cudaSuccess) return e;
  DescLayout dl;  // after the largest accumulator of the batch
  e = desc_layout(smem, dm, false, &dl);
  if (e != cudaSuccess) return e;
  k_deliver_tiled_batch<FMT, ANY><<<n_ctas, kTileThreads, dl.smem, s>>>(nets, bmap, dl.off,
                                                                       dl.cap);
  return cudaGetLastError();
}

cudaError_t launch_deliver_tiled_batch(int fmt, bool any, const BatchNet* nets,
                                       const uint2* bmap, uint32_t n_ctas,
                                       size_t smem, cudaStream_t s) {
  if (n_ctas == 0) return cudaSuccess;
  if (fmt == SNN_W_FP32_12B)
    return any ? launch_batch_t<SNN_W_FP32_12B, true>(nets, bmap, n_ctas, smem, s)
               : launch_batch_t<SNN_W_FP32_12B, false>(nets, bmap, n_ctas, smem, s);
  return any ? launch_batch_t<SNN_W_BF16_8B, true>(nets, bmap, n_ctas, smem, s)
             : launch_batch_t<SNN_W_BF16_8B, false>(nets, bmap, n_ctas, smem, s);
}

uint32_t update_threads() { return kUpdThreads; }

uint32_t serve_threads() { return kTileThreads; }

template <int FMT, bool ANY>
static cudaError_t launch_serve_t(const BatchNet* nets, ServeNet* sn, ServeCtl* ctl,
                                  uint32_t n_nets, uint32_t n_ctas, size_t smem,
                                  unsigned long long spin_limit, cudaStream_t s) {
  static std::atomic<uint32_t> lim[64];
  size_t dm = 0;
  cudaError_t e = allow_tile_smem(k_serve<FMT, ANY>, lim, &dm);
  if (e != cudaSuccess) return e;
  DescLayout dl;  // after the largest accumulator of the nets
  e = desc_layout(smem, dm, false, &dl);
  if (e != cudaSuccess) return e;
  k_serve<FMT, ANY><<<n_ctas, kTileThreads, dl.smem, s>>>(nets, sn, ctl, n_nets, dl.off,
                                                          dl.cap, spin_limit);
  return cudaGetLastError();
}

cudaError_t launch_serve(int fmt, bool any, const BatchNet* nets, ServeNet* sn,
                         ServeCtl* ctl, uint32_t n_nets, uint32_t n_ctas,
                         size_t smem, unsigned long long spin_limit,
                         cudaStream_t s) {
  if (n_nets == 0 || n_ctas == 0) return cudaSuccess;
#define SNN_SERVE(F, ANY) \
  launch_serve_t<F, ANY>(nets, sn, ctl, n_nets, n_ctas, smem, spin_limit, s)
  if (fmt == SNN_W_FP32_12B)
    return any ? SNN_SERVE(SNN_W_FP32_12B, true) : SNN_SERVE(SNN_W_FP32_12B, false);
  return any ? SNN_SERVE(SNN_W_BF16_8B, true) : SNN_SERVE(SNN_W_BF16_8B, false);
#undef SNN_SERVE
}

cudaError_t launch_prepare_external(const NetView& v, const uint32_t* src,
                                    const int32_t* t, uint32_t n,
                                    SpikeEntry* list,
                                    unsigned long long* pair, cudaStream_t s) {
  k_prepare_external<<<1, 1024, 0, s>>>(v, src, t, n, list, pair);
  return cudaGetLastError();
}

}  // namespace snn

// ---------------------------------------------------------------------------
// Allocation-free delivery of a caller's spike list.
//
// snn_deliver stages a caller's list in a buffer the library grows with
// cudaMalloc.  Some callers cannot let a library allocate: processes whose
// device memory is fully reserved by another allocator (a framework's caching
// allocator holding all of HBM), and latency-critical loops where cudaMalloc's
// implicit device synchronisation is not acceptable.  For them the list is
// staged in this file-scope device array instead: a fixed 4 MiB (2^18
// entries) held by every GPU that loads the library until the process exits.
// All calls share it, so calls whose work overlaps on the GPU race; the
// counters that must start at zero are cleared by every call.
// ---------------------------------------------------------------------------
namespace snn {
namespace {
struct NoAllocScratch {
  SpikeEntry list[SNN_NOALLOC_MAX_SPIKES];
  unsigned long long pair;
  unsigned int done;
  unsigned int pad_;
};
static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
NoAllocScratch* g_noalloc_ptr[kMaxDevices] = {};

// Device address of the scratch on the current device, looked up once per
// device (in host code the symbol is only a stand-in for that address).
cudaError_t noalloc_scratch(NoAllocScratch** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = static_cast<NoAllocScratch*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_deliver_noalloc(const NetView& v, const uint32_t* src,
                                   const int32_t* t, uint32_t n,
                                   cudaStream_t s) {
  if (n > SNN_NOALLOC_MAX_SPIKES) return cudaErrorInvalidValue;
  if (deliver_raw_fits(v, n)) return launch_deliver_raw(v, src, t, n, s);
  NoAllocScratch* sc = nullptr;
  cudaError_t e = noalloc_scratch(&sc);
  if (e != cudaSuccess) return e;
  // the list counters must start at zero: clear them on every call
  e = cudaMemsetAsync(&sc->pair, 0, sizeof(unsigned long long) + 2 * sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  e = launch_prepare_external(v, src, t, n, sc->list, &sc->pair, s);
  if (e != cudaSuccess) return e;
  return v.lay != kLayRecords
             ? launch_deliver_tiled(v, &sc->pair, &sc->done, sc->list, n, 0, s)
             : launch_deliver(v, &sc->pair, &sc->done, sc->list, 0, s);
}
}  // namespace snn
