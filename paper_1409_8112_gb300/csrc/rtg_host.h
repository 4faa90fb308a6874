// Host-side internals shared by rtg_api.cu (contexts, builds) and rtg_serve.cu (the request
// server).  Not part of the ABI.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <unordered_map>
#include <vector>

#include "rtg.h"
#include "rtg_internal.cuh"

namespace rtghost {

struct DevBuf {
  void* p = nullptr;
  size_t cap = 0;
  unsigned long long gen = 0;  // allocation number (contents are lost when it changes)
};

// Host tables last copied to a device buffer, so that unchanged tables are not sent again.
struct Upload {
  std::vector<unsigned char> bytes;
  unsigned long long gen = 0;  // DevBuf::gen they were copied to
};

// Launch decisions remembered per shape (sum n, instances, grids, dtype, widest d, flags).
using ShapeKey = std::tuple<long long, int, int, int, int, int, int>;
struct ShapeGuess {
  bool key64 = true;
  int key_bits = 64;
  int cell_bits = 0;  // widest grid's cell index range (bits), the key of a cell-major sort
  long long pair_cap = 0;
  bool sorted_cfg = false;  // sort chosen (tuned or default) for this shape
  rtg::SortConfig sort;
  float cand_per_pos = -1.0f;  // in-cell candidates per sorted position at the last build
  bool pairs_tuned = false;    // enumeration knobs measured for this shape
  int spans_per_warp = 0;      // (tuned) spans per resident warp
  // Kernels left out of the shape's builds (rtg::kSkip* bits), with for each the builds in a row
  // that had nothing for it.  A decision that follows every build changes the launch sequence
  // with every other input near a margin, and each change captures the graph again (60 to 110
  // us): so a kernel that had work comes back at once and goes only after kCalmBuilds.
  int skip = 0;
  int calm[4] = {kCalmBuilds, kCalmBuilds, kCalmBuilds, kCalmBuilds};
  // Builds in a row whose keys needed fewer bits than key_bits / cell_bits hold, and the widest
  // of them (too few bits cost a second build, one pass too many a few per cent).
  int narrow = 0, narrow_key = 0, narrow_cell = 0;
  static constexpr int kCalmBuilds = 16;
  // Builds on 64-bit keys that 32 bits would have held before the shape takes those: each costs
  // about a third more (100k points in 6-D 232 us against 178, 1M 1070 against 790), coming
  // back to 64 bits one more build and a capture (400 us, 1700 us).
  static constexpr int kWideBuilds = 4;

  // After a build: bit `which` (0..3) stands for a kernel that found no work (idle) or some.
  void settle_skip(int which, bool idle) {
    int& n = calm[which];
    if (!idle) {
      n = 0;
      skip &= ~(1 << which);
    } else if (n >= kCalmBuilds || ++n >= kCalmBuilds) {
      skip |= 1 << which;
    }
  }
  // After a build whose keys took kb bits (the widest cell index cb).
  void settle_bits(int kb, int cb, bool first) {
    if (first || kb > key_bits || cb > cell_bits) {
      key_bits = first ? kb : std::max(kb, key_bits);
      cell_bits = first ? cb : std::max(cb, cell_bits);
      narrow = narrow_key = narrow_cell = 0;
    } else if (kb == key_bits && cb == cell_bits) {
      narrow = narrow_key = narrow_cell = 0;
    } else {
      narrow_key = std::max(narrow_key, kb);
      narrow_cell = std::max(narrow_cell, cb);
      if (++narrow >= (key_bits > 32 && narrow_key <= 32 ? kWideBuilds : kCalmBuilds)) {
        key_bits = narrow_key;
        cell_bits = narrow_cell;
        narrow = narrow_key = narrow_cell = 0;
      }
    }
    key64 = key_bits > 32;
  }
  // Pair-buffer entries after a build that emitted e pairs: kept while they hold 6% more than e
  // and no more than four times that (and 2^20, 8 MB), so that inputs of one shape whose pair counts differ
  // neither overflow the buffer (a second enumeration: twice the time on clustered points) nor
  // change the launch sequence.
  static long long tight_pairs(long long e) { return e + e / 16 + 4096; }
  void settle_pairs(long long e) {
    last_pairs = e;
    if (pair_cap < tight_pairs(e) || pair_cap > 4 * tight_pairs(e) + (1 << 20))
      pair_cap = (e + e / 4 + 4096 + 4095) / 4096 * 4096;
  }
  long long last_pairs = -1;  // pairs of the shape's last build (-1: none)
  // A result keeps its column array, so that one follows the pairs and not the pair buffer: room
  // for the most pairs of the shape's recent builds (kCalmBuilds of less than half in a row bring
  // it down), of one size while they differ little, which suits the pool.  The kernels read it
  // from the output slot, so that a change does not change the launch sequence.
  long long col_pairs = -1, sparse_most = 0;
  int sparse = 0;
  void settle_cols(long long e) {
    sparse_most = std::max(sparse_most, e);
    if (e > col_pairs + col_pairs / 32 || (2 * e < col_pairs && ++sparse >= kCalmBuilds)) {
      col_pairs = sparse_most;
    } else if (2 * e < col_pairs) {
      return;
    }
    sparse = 0;
    sparse_most = 0;
  }
  long long col_cap(bool sym) const {
    const long long c = col_pairs < 0 ? pair_cap : std::min(pair_cap, tight_pairs(col_pairs));
    return c * (sym ? 2 : 1);
  }
  // Default brute force: the radius (and form) at which the plan left the pairs to the CUDA cores,
  // and the builds at that radius that keep to them without asking it again.  Operands, plan and
  // the tiles' launch cost 8 to 20 us that such builds wait for (9000 points in 2-D 164 us without,
  // 183 with); points of another extent at the same radius get the tiles kCalmBuilds builds late.
  double no_tiles_r = 0.0;
  bool no_tiles_two_pass = false;
  int no_tiles = 0;
  bool ask_tiles(double r, bool two_pass) const {
    return no_tiles == 0 || r != no_tiles_r || two_pass != no_tiles_two_pass;
  }
  void settle_tiles(bool asked, bool used, double r, bool two_pass) {
    if (!asked) {
      --no_tiles;
    } else {
      no_tiles = used ? 0 : kCalmBuilds;
      no_tiles_r = r;
      no_tiles_two_pass = two_pass;
    }
  }
};

// A result whose columns fill less than half of their array, and leave more than this many entries
// of it unused, is copied to an array of its own size (but for a shape's first).  With four
// fifths for the half, three clustered 50k sets in 9-D in turn took 3407 us a build instead of
// 3262: one of them was copied, 0.4 GB.
constexpr long long kColSlack = 1 << 16;

// A build's launch sequence captured once and replayed for later builds of the same shape.
struct GraphEntry {
  cudaGraphExec_t exec = nullptr;
  std::vector<unsigned char> sig;  // launch arguments it was captured with
  int launches = 0;
};

// Sort variant per (sorted elements, key bits), measured by the autotuner.
using SortKey = std::pair<long long, int>;
struct TuneEntry {
  rtg::SortConfig cfg;
  double us = 0;  // measured time of the sort, microseconds
};

// One build: a batch of instances sharing m, dtype and the points' location.
struct Request {
  const rtg_instance* items;
  int count;
  int m;  // 0: brute force (count must be 1)
  int dtype;
  int points_on_device;
  uint32_t flags;
  bool count_only;
  bool grid_major = false;  // the sorted keys must come out grid by grid (the index reads them so)
};

struct Server;  // request server of a context (rtg_serve.cu)

// Reported pairs per point of recent builds, per d: a decaying maximum (a figure per size
// class of n was measured to correct more first builds, not fewer).
struct PppHints {
  std::map<int, double> h;
  double get(int d) const {
    const auto it = h.find(d);
    return it == h.end() ? 0.0 : it->second;
  }
  void put(int d, double ppp) {
    double& x = h[d];
    x = std::max(0.9 * x, ppp);
  }
  void raise(int d, double ppp) {
    double& x = h[d];
    x = std::max(x, ppp);
  }
};

}  // namespace rtghost

struct rtg_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  uint64_t budget = 0;
  int num_sms = 0;
  std::mutex mu;       // one build at a time
  std::mutex live_mu;  // output bookkeeping (live, out_bytes)
  std::string err;
  rtghost::DevBuf status, inst, iplan, gplan, bases, T64, pts, pf, key_mat, keys0, keys1,
      vals0, vals1, lookback, hist, digit_off, row_cnt, scan_lb, large, large_job, pair_buf,
      tc_tiles, tc_norms, tc_plan, out_slot, sort_epoch, q_idx, q_slots, bits;
  rtg::Status* h_status = nullptr;  // pinned
  rtg::OutSlot* h_slot = nullptr;   // pinned; copied to out_slot before the output kernels
  bool use_graphs = true;           // RTG_GRAPHS=0 launches every kernel directly
  bool cell_major = true;           // RTG_CELL_MAJOR=0 keeps the grid in every sort key
  std::map<rtghost::ShapeKey, rtghost::GraphEntry> graphs;
  cudaMemPool_t pool = nullptr;     // output CSRs (stream ordered, kept cached)
  bool own_pool = true;             // false: a serving lane drawing on its owner's pool
  cudaEvent_t ev[8] = {};
  // the output-slot copy runs on a second stream beside the front of the build
  cudaStream_t side = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  // the optional scratch the running call uses (give_back leaves it)
  bool slots_in_use = false, tiles_in_use = false;
  size_t ws_bytes = 0;
  size_t ws_need = 0;  // workspace bytes the current build asked for (at most ws_bytes)
  size_t out_bytes = 0;
  uint64_t next_handle = 1;
  std::unordered_map<uint64_t, size_t> live;  // CSR handle -> bytes
  std::map<rtghost::ShapeKey, rtghost::ShapeGuess> guesses;
  // Pairs per point of recent builds: the pair-buffer size of a shape built for the first
  // time, so that clustered inputs seldom overflow it.
  rtghost::PppHints ppp_hint;
  std::map<rtghost::SortKey, rtghost::TuneEntry> sort_tune;  // autotuner results
  std::string tune_path;                                     // JSON cache ("" = none)
  std::string device_name;
  bool autotune = true;
  // shapes with more in-cell candidates keep the default enumeration knobs (the trials would
  // each enumerate them all); RTG_TUNE_PAIRS_MAX_CAND
  double tune_pairs_max_cand = 4.0e9;
  bool sort_forced = false;  // RTG_SORT_VARIANT
  rtg::SortConfig sort_force;
  std::vector<rtg::Inst> h_inst;
  std::vector<double> h_T;
  unsigned long long alloc_gen = 0;
  void* h_stage = nullptr;  // pinned staging for the instance and transform tables
  size_t h_stage_cap = 0;
  rtghost::Upload up_inst, up_T;
  rtghost::Server* server = nullptr;  // created by the first rtg_submit
  int last_sorted = 0;  // keys/vals buffer (0 or 1) that holds the last build's sorted keys
  // Width of the keys the last build left there and in key_mat: the width its shape was guessed
  // to need, which stays at 64 bits for a while after a build that needed more than 32.
  bool last_key64 = false;
  // Failure-path hooks (rtg_set_test_hooks): the bounded device waits' iteration limit (0:
  // the default), waits made to wait for something that never happens (rtg::kInject*), and
  // the number of the device allocation that is made to fail (0: none).
  unsigned int spin_limit = 0;
  unsigned int inject = 0;
  long long fail_alloc_at = 0;
  std::atomic<long long> alloc_calls{0};
};

namespace rtghost {

// The status buffer holds the Status counters, then the bounding boxes of the build's
// instances (zeroed together, by one memset, at the start of every build).
constexpr size_t kStatusBytes = (sizeof(rtg::Status) + 255) & ~size_t(255);
inline unsigned long long* bbox_of(rtg_ctx* c) {
  return reinterpret_cast<unsigned long long*>(static_cast<char*>(c->status.p) + kStatusBytes);
}

rtg_status fail(rtg_ctx* ctx, rtg_status s, const std::string& msg);
std::string& last_error_text();
// Output memory of ctx's pool, ordered on stream s; counted in ctx's out_bytes.
rtg_status alloc_out_on(rtg_ctx* ctx, cudaStream_t s, size_t bytes, void** p);
uint64_t register_out(rtg_ctx* ctx, size_t bytes);
void release_out(rtg_ctx* ctx, rtg_csr* csr);
rtg_status validate_common(int dtype, int64_t n, int d, double r, double c, const void* points);
rtg_status validate_transforms(const double* T, int d, int m);
rtg_status build(rtg_ctx* c, const Request& q, rtg_csr* out);
// A context of the same device with its own stream, workspace and pool (no server).
rtg_status create_ctx(int device, uint64_t budget, void* stream, rtg_ctx** out);
void destroy_ctx(rtg_ctx* c);
// Frees the per-build workspace (points, rows, keys, pair buffer, ...), the captured graphs and
// the output pool's cached blocks; the next build allocates again.  The caller holds c->mu.
void trim_workspace(rtg_ctx* c);
void stop_server(rtg_ctx* c);  // joins the server's threads; frees unclaimed results
void notify_server(rtg_ctx* c);  // memory was released: waiting requests are considered again

// Sort autotuner (rtg_tune.cu).
// The variant used without measurement: 8-bit digits, 2048-key tiles, look-back while the
// tiles fit in about three waves.
rtg::SortConfig sort_default(long long N, int num_sms);
// Sorts the keys of `a` (regenerated by the key kernel before every trial) with every compiled
// variant and strategy, five times, and returns the one with the lowest median time; records
// it in the context's table and JSON cache.  Needs a's buffers sized for any variant.
rtg_status tune_sort(rtg_ctx* c, rtg::BuildArgs& a, long long N, int key_bits,
                     rtg::SortConfig* out);
// Times the in-cell enumeration of a's keys (sorted with cfg) for each spans-per-warp candidate
// and returns the fastest; 0 (the default) when a first trial takes long.
rtg_status tune_pairs(rtg_ctx* c, rtg::BuildArgs& a, const rtg::SortConfig& cfg, int key_bits,
                      int* spans_per_warp);
size_t sort_scratch_bytes(long long N, const rtg::SortConfig& cfg);  // look-back / counts
size_t sort_scratch_bytes_max(long long N);
void tune_load(rtg_ctx* c);

// Workspace and status helpers (rtg_api.cu).
void free_buf(rtg_ctx* c, DevBuf& b);
// alloc_out_on(c, c->stream, ...), tried again without the optional scratch.  The caller holds c->mu.
rtg_status alloc_out(rtg_ctx* c, size_t bytes, void** p);
rtg_status ensure(rtg_ctx* c, DevBuf& b, size_t bytes, bool zero = false);
rtg_status read_status(rtg_ctx* c);
rtg_status check_errors(rtg_ctx* c, unsigned int mask);
// Grid parameters for a target recall (rtg_params.cu).
rtg_status tune_params(rtg_ctx* c, const void* points, int dtype, int on_device, int64_t n, int d,
                       double r, double target, uint64_t seed, uint32_t flags,
                       rtg_param_choice* out);
// Neighbour lists of a subset of the points from a symmetric CSR (rtg_query.cu).
rtg_status query_neighbors(rtg_ctx* c, const rtg_csr* g, const int32_t* queries, int64_t nq,
                           int queries_on_device, rtg_csr* out);
rtg_status index_create(rtg_ctx* ctx, const rtg_instance& it, int m, int dtype, int on_device,
                        rtg_index** out);
rtg_status index_query(rtg_ctx* ctx, const rtg_index* ix, const void* queries, int on_device,
                       int64_t nq, rtg_csr* out);
void index_destroy(rtg_ctx* ctx, rtg_index* ix);

}  // namespace rtghost
