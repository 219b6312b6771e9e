// snn_net.cuh -- host-side definition of a net (shared by the C ABI and the
// serving loop).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>
#include <math.h>

#include "snn_internal.cuh"

using namespace snn;

namespace snn {
// Message returned by snn_last_error() on this thread.
void set_last_error(const char* msg);
// Tile geometry the store builder uses for n targets (see snn_api.cu).
void tile_geometry(uint32_t n, int window, int32_t hint, uint32_t* tile_w,
                   int* lo_bits, uint32_t* n_tiles);
// Device memory from the library's stream-ordered pool of the current
// device (see snn_api.cu); free with pool_free on a stream ordered after
// the last use.
cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s);
void pool_free(void* p, cudaStream_t s);
// Keep (+1) or let go (-1) of the device's pool: while held, memory freed by
// destroyed nets stays in the pool for the next ones (a server holds it for
// its lifetime, so that admitting a request never waits for memory to be
// mapped again).
void pool_hold(int dev, int delta);
// snn_simulate's asynchronous production path (serving uses it directly:
// may_capture false keeps it from instantiating a graph while builds run).
int simulate_async(snn_net* net, int64_t n_steps, bool may_capture);
}  // namespace snn

// The net: parameters, device buffers and host bookkeeping.
struct snn_net {
  snn_params p{};
  cudaStream_t stream = nullptr;
  bool counted = false;  // counted among the device's live nets
  bool own_stream = false;
  int device = 0;
  uint32_t n = 0, pitch = 0;
  uint32_t n_src = 0, g0 = 0;  // store rows (all sources); first neuron
  int fmt = 0, n_slots = 0;
  UpdConst uc{};
  float *V = nullptr, *I = nullptr, *J = nullptr;
  int32_t* refr = nullptr;
  float* rb = nullptr;
  uint32_t* counts = nullptr;
  Ctl* ctl = nullptr;
  uint64_t* row_ptr = nullptr;
  void* recs = nullptr;
  uint64_t n_syn = 0, recs_bytes = 0;
  uint64_t n_pad = 0;            // records the store has room for
  int lay = kLayRecords, d_base = 0;
  bool int_w = false;            // weights fit 16-bit integers (kLayI16)
  bool hom = false;              // uniform weights (kLayHom if tiled)
  uint32_t hom_split = 0;
  float hom_w[2] = {0.f, 0.f};
  uint32_t* tile_off = nullptr;  // [n][n_tiles + 1]
  bool check_noted = false;      // SNN_ERRF_CHECK counted (checked builds)
  uint32_t* xbuf = nullptr;      // caller's exchange buffer (snn_set_exchange)
  uint32_t xcap = 0;
  const void* x_parts_ok = nullptr;  // last gathered-parts pointer validated
  uint32_t tile_w = 0, n_tiles = 0;
  uint32_t pl_tiles = 0, tile_grp = 1;  // see NetView
  int lo_bits = 0;
  int window = 0;
  uint32_t mult_max = 0, k_in_max = 0, spikes_per_iv = 1;
  int own_mode = kAddAny;  // own_add_mode, from snn_finalize on
  int acc_words = 2, acc_qs_min = 0;  // accumulator cells (see NetView)
  float max_abs_w = 0.f;
  SpikeEntry* list = nullptr;
  uint64_t list_cap = 0;
  unsigned long long* sim_flags = nullptr;  // see SimShared
  int cycle_max = kCycleMax;                // snn_set_cycle
  uint32_t sim_polls = kSimPolls;           // snn_debug_cycle
  bool sim_unscaled = false, sim_refused = false;
  SpikeEntry* ext_list = nullptr;
  uint32_t* ext_src = nullptr;
  int32_t* ext_t = nullptr;
  uint64_t ext_cap = 0;
  uint32_t* log_src = nullptr;
  int32_t* log_t = nullptr;
  uint64_t log_cap = 0;
  bool connected = false, finalized = false, pending = false;
  int interval = 0, dmin = 0, dmax = 0;
  long long t_host = 0;
  bool profiling = false;
  std::vector<cudaEvent_t> ev;
  double ms_update = 0, ms_deliver = 0;
  uint64_t launches = 0, upd_launches = 0, del_launches = 0;
  cudaGraphExec_t graph = nullptr;
  cudaGraphExec_t graph_prof = nullptr;  // the same intervals with timing events
  // STDP (snn_set_stdp): parameters and device state (StdpView)
  bool stdp_on = false;
  snn_stdp_params stdp{};
  StdpView sp{};
  // long-run spike statistics
  int32_t* isi_last = nullptr;
  uint32_t* isi_spikes = nullptr;
  uint32_t* isi_n = nullptr;
  double* isi_sum = nullptr;
  double* isi_sq = nullptr;

  // Lanes per run (2^lg) from the mean run of a tile (in synapses) and the number
  // of rows.  A lane has three 16-byte vectors loaded ahead (8 cells, or 4 joined
  // words or weights) and every group of 32 / lanes runs costs a fixed number of
  // instructions; runs past what is ahead want more lanes, and so do rows that lie
  // far apart, of which a warp's request then touches fewer: the first lines sit
  // at run x sqrt(rows).  Measured where two numbers of lanes take the same time
  // (deliveries of 1,400 and 3,000 spikes; 20,003, 60,000 and 112,500 neurons):
  //             1 | 2      2 | 4 lanes                4 | 8       8 | 16  16 | 32
  //   cells     9-10       26, 17, 12                 92          310     500
  //   words     3.5        16, 5.5, 5                 47          110     235
  //   FP32      3          11, 4.5, 4.5               22, 11.5, 9.5  90   320
  // (500: extrapolated.)  Either side, 3,000 spikes, 60,000 neurons, us: cells 74
  // on 4 lanes 38.3, on 8 40.8, 120 52.4, 50.5; words 37 28.5, 32.4, 60 41.1, 36.8;
  // FP32 9 33.9, 38.0, 20 50.1, 40.4, 37 73.1, 48.8.  Words between 5.5 and 16 are a
  // compromise: 13 on 20,003 neurons take 19.2 us on 2 lanes and 21.2 on 4, but the
  // shorter lists of their one-launch cycle 1,428 and 1,378 us for 100 intervals.
  // In that cycle (a few hundred spikes, rows already in L2) 8 lanes pay earlier,
  // us an interval on 4 and 8: words 20 12.4, 12.8, 37 17.0, 15.8; cells (BF16) 30
  // 16.2, 16.9, 40 16.5, 16.2, 50 17.0, 16.2, 74 28.6, 27.8, (FP32) 60 16.2, 16.3.
  void set_layout(NetView* v) const {
    v->lay = lay;
    v->d_base = d_base;
    v->hom_split = hom_split;
    v->hom_w[0] = hom_w[0];
    v->hom_w[1] = hom_w[1];
    v->dat = recs;
    v->cells = nullptr;
    v->tgts = nullptr;
    v->row_mul = 1;
#if SNN_CHECK
    v->n_pad = n_pad;
#endif
    v->lg = v->lg_cycle = 0;
    v->mean_row = n_src ? (float)((double)n_syn / n_src) : 0.f;
    if (lay == kLayRecords) return;
    if (fmt == SNN_W_FP32_12B) {
      const char* p = static_cast<const char*>(recs);
      v->tgts = reinterpret_cast<const uint32_t*>(p + 4 * n_pad);
      v->cells = reinterpret_cast<const uint16_t*>(p + 8 * n_pad);
      if (lay == kLayHom) v->dat = v->cells;
    } else {
      v->row_mul = lay == kLayHom ? 4 : 2;
    }
    const double run =
        n_src && n_tiles ? (double)n_syn / ((double)n_src * n_tiles) : 0.0;
    v->lg = run_lanes(run, 0);
    v->lg_cycle = run_lanes(run, 1);
  }
  int run_lanes(double run, int cycle) const {
    const int k = lay == kLayHom ? 0 : lay == kLayF32 ? 2 : 1;
    static const double first[3] = {9.5, 3.5, 3.0}, far_apart[3] = {4000, 1750, 1350};
    static const double eight[2][2] = {{92, 47}, {45, 26}};
    static const double more[3][2] = {{310, 500}, {110, 235}, {90, 320}};
    const double spread = run * sqrt((double)n_src);
    if (run < first[k]) return 0;
    if (spread < far_apart[k]) return 1;
    if (k == 2 ? spread < 3000.0 : run < eight[cycle][k]) return 2;
    return run < more[k][0] ? 3 : run < more[k][1] ? 4 : 5;
  }

  NetView view() const {
    NetView v;
    v.n = n;
    v.n_src = n_src;
    v.g0 = g0;
    v.pitch = pitch;
    v.slot_mask = (uint32_t)n_slots - 1u;
    v.chunk = (uint32_t)chunk_records(fmt);
    v.fmt = fmt;
    v.V = V;
    v.I = I;
    v.J = J;
    v.refr = refr;
    v.rb = rb;
    v.counts = counts;
    v.row_ptr = row_ptr;
    v.recs = recs;
    v.tile_off = tile_off;
    v.tile_w = tile_w;
    v.n_tiles = n_tiles;
    v.pl_tiles = pl_tiles ? pl_tiles : n_tiles;
    v.tile_grp = tile_grp ? tile_grp : 1u;
    v.d_min = dmin;
    v.d_max = dmax;
    v.window = window;
    v.mult_max = mult_max;
    v.k_in_max = k_in_max;
    v.spikes_per_iv = spikes_per_iv;
    v.max_abs_w = max_abs_w;
    v.acc_words = acc_words;
    v.acc_qs_min = acc_qs_min;
    set_layout(&v);
    v.list = list;
    v.list_cap = list_cap;
    v.xbuf = xbuf;
    v.xcap = xcap;
    v.gx = nullptr;
    v.gx_parts = 0;
    v.gx_stride = 0;
    v.gx_cap = 0;
    v.ext_src = nullptr;
    v.ext_t = nullptr;
    v.ext_n = 0;
    v.log_src = log_src;
    v.log_t = log_t;
    v.log_cap = log_cap;
    v.ctl = ctl;
    v.plastic = stdp_on && sp.wp != nullptr;
    v.sp = sp;
    v.isi_last = isi_last;
    v.isi_spikes = isi_spikes;
    v.isi_n = isi_n;
    v.isi_sum = isi_sum;
    v.isi_sq = isi_sq;
    v.own_mode = own_mode;
    return v;
  }
};

