// The library context (opaque at the ABI): host mesh, workspace layout, bound
// device state and the driver.  Shared by api.cpp and adjoint.cpp.
#pragma once

#include <cuda_runtime_api.h>

#include <array>
#include <functional>
#include <string>
#include <vector>

#include "lbm_internal.h"

namespace lbm {
// Ops of the recursive level step, in the order lbm_ctx::advance issues them.
enum StepOp { OP_GFF = 0, OP_MOM_A = 1, OP_GFC_A = 2, OP_SC = 3, OP_MOM_B = 4, OP_GFC_B = 5 };
// Instants that advance at most this many fluid elements launch their kernels
// as programmatic dependents of one another (let_next_start in kernels.cuh).
// Below it the step is a chain of latencies and hiding a launch pays; beyond
// it the waiting blocks take slots that the interior bricks' kernel, beside
// the chain, could use.  Measured per coarse step, chained / not: four-level
// D2Q9 cylinder (6e4 elements) 56 / 67 us, two-level D3Q27 (9e5) 131 / 139 us,
// four-level BF16 sphere (3.6e6) 866 / 857 us.  FP64: a kernel takes as long
// as the SM with the most of its one-warp blocks, and dependents start where
// slots happen to be free, not evenly: 1,800 elements 43.5 / 46.5 us, but
// 4.6e4 elements 60 / 40 us; the line is where every SM has about one warp.
constexpr int64_t kChainElements = 1 << 20, kChainElements64 = 1 << 12;
// Instants of at most this many elements run all interior bricks beside the
// GhostFromCoarser fill (us per coarse step, beside / after: cylinder 54.5 /
// 57.3, two-level 64^3 44.9 / 45.7, D3Q27 9e5 elements 131 / 132; four-level
// sphere of 3.6e6 elements BF16 915 / 750, FP32 1022 / 992, two-level 160^3 372 /
// 367; the sphere of 1.1e7 elements took 7.4 against 4.94 ms).
constexpr int64_t kBesideElements = 1 << 20;
// Graphs of meshes within kBesideElements give the chain of fills and the rest
// one level of priority more than the interior bricks: its blocks, on the
// critical path, start before the waiting bricks' (two-level 64^3 FP32 7450 ->
// 6730 us for 200 steps, D3Q27 96x80x64 4408 -> 4366 for 50; others within
// 0.5%).  Beyond it the mixture slows the bricks (sphere of 1.1e7 elements 4.97
// -> 5.38 ms a step).  The bricks keep the bound stream's priority, so that the
// steps never pass a stream that the caller ranks above it; on a stream of the
// greatest priority all kernels have that one.  (The least and the greatest
// priority of the device instead: 6728 us.)
struct StepPriority {
  int bricks, chain;
};
inline StepPriority step_priority(int bound, int greatest) { return {bound, bound > greatest ? bound - 1 : bound}; }
//
// A graph launch costs about 3.5 us between two replays, 4 to 5% of a step of a
// small mesh with two steps a graph.  Once a context has replayed
// kLongGraphAfter steps (so that a short run pays for no longer capture) and
// has at most kLongGraphUpdates updates a coarse step, it replays graphs of
// kLongGraphSteps: us per call, with its output, D2Q9 channel FP64, 50 steps
// 2003 -> 1879, cylinder, 50 steps 2745 -> 2601, two-level 64^3, 200 steps 8870
// -> 8620, D2Q9 32x32 FP64, 20 steps 811 -> 792.  A step of many instants is
// long against the gap, and its graph large: kLongGraphInstants instants a step
// (five levels, or three in diffusive scaling) keep a long graph to about a
// thousand nodes.  (16 steps in FP32, a long graph against short ones: 16
// instants 1.33 / 1.35 ms, 64 instants 3.02 / 3.04 ms, 1,024 instants, six
// levels in diffusive scaling, 55 / 50 ms and 240 ms to make its 4.1e4 nodes.)
constexpr int kLongGraphSteps = 16;
constexpr int64_t kLongGraphAfter = 64, kLongGraphUpdates = 1 << 21, kLongGraphInstants = 16;
// Kernel kinds of the per-launch timing (lbm_timing_read row kTimedKinds * L + kind)
enum TimedKind { TK_INTERIOR = 0, TK_LIST = 1, TK_BOUNDARY = 2, TK_GFF = 3, TK_MOM = 4, TK_GFC = 5, TK_OUTLET = 6,
                 TK_SC_SPAN = 7 };
constexpr int kTimedKinds = 8;

struct LevelDev {
  size_t gff_child0 = 0, gfc_src = 0, gfc_oct = 0, src_elem = 0, gsrc_elem = 0, gsrc_rec = 0;
  // source records of the two pdf buffers: momA[parity] those of the current
  // state (a stream-collide writes those of its new state into the other one
  // while the GhostFromCoarser fill may still read these)
  size_t momA[2] = {0, 0};
  int64_t nsrc = 0, n_gsrc = 0, n_gsrc_inner = 0;
};

}  // namespace lbm

struct lbm_ctx {
  lbm_params p{};
  lbm::HostMesh M;
  const lbm::Ops* ops = nullptr;
  std::string err;
  int d = 2, Q = 9, nS = 3, nlev = 1;
  double rho_off = 0.0;
  double inlet[lbm::kQmax] = {};
  // layout (byte offsets into the workspace)
  size_t oA = 0, oB = 0, oNbr = 0, oBrickNb = 0, oBrickTab = 0, oInletS = 0, oOutQ = 0, oObsA = 0, oObsQ = 0, oF = 0, oOutElem = 0, oOutA = 0, oOutB = 0, oOutDir = 0, oOutKind = 0,
         oSide = 0, oObsElem = 0, oObsDir = 0, oUslot = 0, oUlev = 0, oSlotUser = 0, oStage = 0, oPartial = 0, oRed = 0,
         oSrcMask = 0, oSrcFirst = 0;
  std::vector<lbm::LevelDev> ld;
  size_t bytes = 0;
  int64_t chunk = 0;
  // bound state
  bool bound = false;
  char* ws = nullptr;
  cudaStream_t st = nullptr;
  std::vector<int> parity;
  // per level, built by the first lbm_adjoint (build_source_lists)
  struct SourceLists {
    std::vector<int32_t> off, item, saved;
  };
  std::vector<SourceLists> source_lists;
  // the two buffers of every level's state, by parity: A and B of the
  // workspace, except while the adjoint records steps into its tape
  std::vector<std::array<void*, 2>> state;
  void reset_state_buffers() { state.assign(nlev, {at(oA), at(oB)}); }
  // recording (adjoint): where a level's next stream-collide writes its new
  // state; and called when the fill at t + 1/2 reads a level's records at t + 1
  std::function<void*(int level)> new_state;
  std::function<void(int level)> at_mid_step;
  // level kernels (lbm_kernel_launches) and the launches that carried them (lbm_launches)
  int64_t launches = 0, issued = 0;
  // optional mass check (params.check_every): coarse steps since the last
  // check, and the reference mass (taken at the first lbm_step after bind,
  // init or set_state)
  int64_t steps_since_check = 0;
  bool mass_ref_valid = false;
  double mass_ref = 0.0;
  int64_t steps_done = 0;  // coarse steps since bind / init / set_state (for messages)
  void reset_check() {
    steps_since_check = 0;
    mass_ref_valid = false;
    steps_done = 0;
    recs_valid = false;
  }
  // the source records momA[parity] of every level hold the moments of the
  // current state (kept by the stream-collide epilogue from one step to the
  // next); cleared by anything else that changes the state, the force or the
  // relaxation rates, and restored by ensure_records()
  bool recs_valid = false;
  void ensure_records();
  // observer called before every op of advance() (records the adjoint tape);
  // with dry set, advance() only walks the op sequence and flips parities
  std::function<void(int op, int level)> hook;
  bool dry = false;
  // per-launch timing: 0 off; 1 every kernel of the step, launched kernel by
  // kernel; 2 steps keep replaying the captured graphs, which then record
  // events around the finest level's stream-collide launches
  int timing = 0;
  bool capturing = false;
  struct Timed {
    int li, kernel;  // lbm::TimedKind
    cudaEvent_t a, b;
  };
  std::vector<Timed> timed;
  std::vector<cudaEvent_t> event_pool;
  cudaEvent_t get_event() {
    if (!event_pool.empty()) {
      cudaEvent_t e = event_pool.back();
      event_pool.pop_back();
      return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
  }
  // runs launch(), bracketed by events on stream s (default: the bound
  // stream) when the timing mode asks for this launch
  template <class F>
  void timed_launch(int li, int kind, F&& launch, cudaStream_t s = nullptr) {
    const bool finest_sc = li == nlev - 1 && (kind <= lbm::TK_BOUNDARY || kind == lbm::TK_SC_SPAN);
    const bool rec = (timing == 1 && kind != lbm::TK_SC_SPAN) || (timing == 2 && capturing && finest_sc);
    if (!rec) {
      launch();
      return;
    }
    if (!s) s = st;
    Timed t{li, kind, get_event(), get_event()};
    // inside a capture, only an external record becomes an event-record node
    // of the graph (a plain record would just order the captured work)
    const unsigned flags = capturing ? cudaEventRecordExternal : cudaEventRecordDefault;
    cudaEventRecordWithFlags(t.a, s, flags);
    launch();
    cudaEventRecordWithFlags(t.b, s, flags);
    timed.push_back(t);
  }
  void recycle_timed() {
    for (auto& t : timed) {
      event_pool.push_back(t.a);
      event_pool.push_back(t.b);
    }
    timed.clear();
  }
  // CUDA graphs of two coarse steps (every level's A/B parity is back where it
  // started after two coarse steps) or of one, per starting parity state;
  // kernel arguments are baked in, so any change of them drops the graphs
  struct StepGraph {
    std::vector<int> parity;  // at the start
    std::vector<int> end;     // after the replay
    int steps;
    cudaGraphExec_t exec;
    int64_t launches, issued;
    std::vector<Timed> timed;  // event pairs recorded by the graph (timing mode 2)
  };
  std::vector<StepGraph> graphs;
  cudaStream_t cap_stream = nullptr;
  // of the kernels in the captured steps (lbm_bind: by the bound stream's)
  lbm::StepPriority prio{0, 0};
  void set_priority();
  // branch streams and fork/join events of the captured graphs: [0] the
  // interior bricks, [1] the boundary values
  struct Branches {
    cudaStream_t s[2] = {nullptr, nullptr};
    cudaEvent_t fork[2] = {nullptr, nullptr}, join[2] = {nullptr, nullptr};
    bool ok = false;
  } br;
  bool make_branches();
  // copy stream of lbm_init's double-buffered host uploads: copy_ev[0..1]
  // mark each staging half free again, [2] the bound stream's earlier work,
  // [3] a half-chunk's copies done (made on first use; false if unavailable)
  cudaStream_t copy_st = nullptr;
  cudaEvent_t copy_ev[4] = {nullptr, nullptr, nullptr, nullptr};
  bool copy_tried = false;
  bool copy_stream_ready() {
    if (!copy_tried) {
      copy_tried = true;
      bool ok = cudaStreamCreateWithFlags(&copy_st, cudaStreamNonBlocking) == cudaSuccess;
      for (cudaEvent_t& e : copy_ev) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
      if (!ok) {
        cudaGetLastError();
        if (copy_st) cudaStreamDestroy(copy_st);
        for (cudaEvent_t& e : copy_ev)
          if (e) cudaEventDestroy(e);
        copy_st = nullptr;
        for (cudaEvent_t& e : copy_ev) e = nullptr;
      }
    }
    return copy_st != nullptr;
  }
  bool prioritised() const {
    int64_t n = 0;
    for (const lbm::HostLevel& H : M.lv) n += H.nF;
    return n <= lbm::kBesideElements;
  }
  // 64 bytes of pinned host memory that kernels can write (made by lbm_bind;
  // null if unavailable)
  double* result_host = nullptr;
  bool result_tried = false;
  double* pinned_result() {
    if (!result_tried) {
      result_tried = true;
      void* q = nullptr;
      if (cudaHostAlloc(&q, 64, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) result_host = static_cast<double*>(q);
      else cudaGetLastError();
    }
    return result_host;
  }
  bool graphs_on = true;
  bool long_graphs_on = true;  // false once a long graph could not be made
  int64_t graph_steps = 0;     // replayed since the graphs were last dropped
  bool long_graphs() const {
    int64_t updates = 0, instants = 1;
    for (int li = 0; li < n_filled; ++li) {
      if (li) instants *= lbm::time_ratio(p.time_mode);
      updates += M.lv[li].nF * instants;
    }
    return long_graphs_on && timing == 0 && graph_steps >= lbm::kLongGraphAfter && updates <= lbm::kLongGraphUpdates &&
           instants <= lbm::kLongGraphInstants;
  }
  int last_graph = -1;        // graph of the most recent replay
  bool graph_unread = false;  // its events hold a replay not yet read
  void drop_graphs() {
    for (auto& g : graphs) {
      cudaGraphExecDestroy(g.exec);
      for (auto& t : g.timed) {
        event_pool.push_back(t.a);
        event_pool.push_back(t.b);
      }
    }
    graphs.clear();
    graph_steps = 0;
    last_graph = -1;
    graph_unread = false;
  }
  ~lbm_ctx() {
    drop_graphs();
    recycle_timed();
    for (cudaEvent_t e : event_pool) cudaEventDestroy(e);
    drop_streams();
    if (result_host) cudaFreeHost(result_host);
    if (copy_st) cudaStreamDestroy(copy_st);
    for (cudaEvent_t e : copy_ev)
      if (e) cudaEventDestroy(e);
  }
  // the capture and branch streams, made again when they are next needed
  void drop_streams() {
    if (cap_stream) cudaStreamDestroy(cap_stream);
    cap_stream = nullptr;
    for (int b = 0; b < 2; ++b) {
      if (br.s[b]) cudaStreamDestroy(br.s[b]);
      for (cudaEvent_t e : {br.fork[b], br.join[b]})
        if (e) cudaEventDestroy(e);
    }
    br = Branches{};
  }

  template <class T = void>
  T* at(size_t off) const {
    return reinterpret_cast<T*>(ws + off);
  }
  void* cur(int li) const { return state[li][parity[li]]; }
  void* nxt(int li) const { return state[li][parity[li] ^ 1]; }
  uint32_t parity_mask() const {
    uint32_t m = 0;
    for (int li = 0; li < nlev; ++li) m |= (uint32_t)(parity[li] & 1) << li;
    return m;
  }
  const void* force_ptr() const { return p.use_force ? at(oF) : nullptr; }

  lbm_status fail(lbm_status s, const std::string& m) {
    err = m;
    return s;
  }
  lbm_status cuda_check(cudaError_t e, const char* where) {
    if (e == cudaSuccess) return LBM_OK;
    err = std::string(where) + ": " + cudaGetErrorString(e);
    return LBM_ERR_CUDA;
  }
  lbm_status launched(const char* where) { return cuda_check(cudaGetLastError(), where); }

  void layout();
  // driver pieces: launch arguments of a level's part of an op, added to
  // those of the levels that share the launch
  lbm::GffArgs gff_args() const;
  void add_gff(lbm::GffArgs& a, int li) const;
  lbm::GfcArgs gfc_args() const;
  // two_times: the fill at t + 1/2; all_layers false: in LINEAR mode the outer
  // ghost layer, which no stream-collide reads, is left unwritten
  void add_gfc(lbm::GfcArgs& a, int li_fine, bool two_times, bool all_layers) const;
  lbm::OutletArgs outlet_args(const void* side) const;
  void add_outlet(lbm::OutletArgs& o, int li, const void* src) const;
  lbm::ScArgs sc_args() const;
  // elements of one kind (TK_INTERIOR, TK_BOUNDARY, TK_LIST) of level li as a
  // segment, the level in slot `slot`; returns 1 if there are any, else 0
  int add_sc(lbm::ScArgs& a, int slot, int li, int kind) const;
  lbm::SourceTable source_table() const;
  template <class Args>
  void ghost_units(Args& a, bool to_coarse) const;
  // ops of one level, on the bound stream
  void fill_gff(int li);
  // records of the level's sources into mom_off: subset SRC_ALL every source,
  // SRC_GFF_OUTER the ghosts of the outer GhostFromFiner layer
  void source_moments(int li, size_t mom_off, cudaStream_t s = nullptr, int subset = 0);
  enum { SRC_ALL = 0, SRC_GFF_OUTER = 1 };
  void fill_gfc(int li_fine, bool two_times, bool all_layers);
  void stream_collide(int li);
  // one coarse step, the levels batched by instant (a graph capture, or
  // launched at once where the adjoint records it)
  void step_batched();
  bool can_batch() { return n_filled <= lbm::kMaxBatch && make_branches(); }
  void tick_batched(int l0, int n);
  int n_filled = 1;                  // levels up to the finest one with elements
  bool outlet_reads_ghosts = false;  // a boundary value reads a ghost's pdfs
  // one coarse step, level by level
  void advance(int li);
  // one coarse step from the top: ensure_records(), then advance(0)
  void coarse_step() {
    ensure_records();
    advance(0);
  }
  // graph of nsteps (1, or an even number) coarse steps from the current parity state,
  // captured on first use; null when capture is unavailable: the caller steps
  // eagerly (graphs_on cleared) or, of a long graph, with shorter ones
  // (long_graphs_on cleared)
  const StepGraph* step_graph(int nsteps);
  // n coarse steps as lbm_step issues them (graph replay unless timing mode 1)
  lbm_status run_steps(int64_t n_coarse);
};

