// Discrete adjoint driver: checkpointed reverse sweep over the multilevel step.
//
// lbm_adjoint runs the forward steps from the current state, keeping a copy of
// the state every K coarse steps.  Going backwards segment by segment, it
// records the segment's steps: the stream-collides write every new state into
// a tape of states instead of the two buffers, so that the reverse reads them
// in place, nothing copied.  Either the whole segment is recorded at once (the
// last one already while the forward passes through it), or each step, last to
// first, from its starting state.  The reverse kernels then run the steps' ops
// in the reverse of the recursive order.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "lbm_ctx.h"
#include "lbm_internal.h"

using namespace lbm;

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct TapeOp {
  int op = 0, level = 0;
  int k = 0;   // state the op reads, of its level (GFF: of the finer level; GFC: records at t of the coarser
               // level): 0 the step's start, k the one its k-th stream-collide in the step wrote
  int kb = 0;  // GFC B: state of the records at t + 1
  int mid = 0; // MOM B, GFC B: how many of the level's mid-step saves precede the op's
  std::vector<int> parity;  // parities of all levels before the op
};

struct AdjLayout {
  size_t lamA = 0, lamB = 0, lamF = 0, side_fwd = 0, lam_side = 0, partial = 0, acc = 0, contrib = 0;
  std::vector<size_t> lam_rec, recA, recB, csr_off, csr_item;
  std::vector<size_t> src_saved;  // per level: index of each record among the saved sources, or -1
  std::vector<size_t> save_off, save_bytes;  // per level: its saves in a step's part of the tape
  size_t ck = 0, steps = 0, tape = 0, fin = 0;
  int n_ck = 0, n_steps = 0;
  int n_slots = 0;        // states of the most often advanced level in one coarse step
  bool tape_all = false;  // a whole segment on the tape, else one step
  size_t state_bytes = 0, step_bytes = 0, total = 0;
  int partial_rows = 0;  // running rows of the parameter sums: the largest grid of a reverse launch
  int side_row0 = 0;     // first row of the neighbour-list reverse, which runs beside the brick reverse
};

// Copies the rows of level li's segment of a [Q][Ntot] state.
void copy_level(lbm_ctx* c, const void* from, void* to, int li) {
  const HostLevel& H = c->M.lv[li];
  const size_t s = c->ops->storage_bytes;
  launch_copy_rows(from, to, (size_t)c->M.Ntot * s, (size_t)H.base * s, (size_t)H.N * s, c->Q, s, c->st);
}

// The ops of one coarse step in the order of the recursion (a dry walk from
// the current parities, launching nothing): the reverse sweep's program.
std::vector<TapeOp> plan_step(lbm_ctx* c) {
  std::vector<TapeOp> tape;
  std::vector<int> sc(c->nlev, 0), at_a(c->nlev, 0), mids(c->nlev, 0);
  const std::vector<int> saved = c->parity;
  c->hook = [&](int op, int li) {
    TapeOp t;
    t.op = op;
    t.level = li;
    t.parity = c->parity;
    switch (op) {
      case OP_GFF: t.k = sc[li + 1]; break;
      case OP_MOM_A: t.k = at_a[li] = sc[li]; break;
      case OP_GFC_A: t.k = at_a[li - 1]; break;
      case OP_SC: t.k = sc[li]++; break;
      case OP_MOM_B:
        t.k = sc[li];
        t.mid = mids[li]++;
        break;
      case OP_GFC_B:
        t.k = at_a[li - 1];
        t.kb = sc[li - 1];
        t.mid = mids[li - 1] - 1;
        break;
    }
    tape.push_back(t);
  };
  c->dry = true;
  c->advance(0);
  c->dry = false;
  c->hook = nullptr;
  c->parity = saved;
  return tape;
}

// One recorded coarse step: per level its states in the step (the start, then
// one per stream-collide), and the GhostFromFiner sources' pdfs at the end of
// each of its substeps, which the next GhostFromFiner fill overwrites in place
// (LINEAR mode: the records at t + 1 include them).
struct Recorded {
  std::vector<std::vector<const void*>> states, mids;
  const void* state(int li, int k) const { return k < (int)states[li].size() ? states[li][k] : nullptr; }
  const void* mid(int li, int k) const { return k < (int)mids[li].size() ? mids[li][k] : nullptr; }
};

// substeps of level li in a coarse step
int64_t substeps(const lbm_ctx* c, int li) {
  int64_t n = 1;
  for (int l = 0; l < li; ++l) n *= time_ratio(c->p.time_mode);
  return n;
}

const AdjOps* adj_ops_for(int precision) {
  if (precision == LBM_FP64) return adj_ops_fp64();
  if (precision == LBM_FP32DEV) return adj_ops_fp32dev();
  return adj_ops_bf16dev();
}

AdjLayout adj_layout(lbm_ctx* c, int64_t n, int K) {
  AdjLayout L;
  size_t o = 0;
  auto take = [&](size_t b) {
    size_t r = o;
    o += align_up(std::max<size_t>(b, 1));
    return r;
  };
  const size_t N = (size_t)c->M.Ntot;
  const size_t lb = c->p.precision == LBM_FP64 ? 8 : 4;
  L.lamA = take(c->Q * N * lb);
  L.lamB = take(c->Q * N * lb);
  L.lamF = take((size_t)c->d * N * 8);
  L.side_fwd = take(c->M.out_elem.size() * lb);
  L.lam_side = take(c->M.out_elem.size() * lb);
  const AdjOps* aops = adj_ops_for(c->p.precision);
  const int64_t block = aops->sc_block;
  int64_t interior = 1, rest = 0;
  for (int li = 0; li < c->nlev; ++li) {
    const HostLevel& H = c->M.lv[li];
    // four lanes a source at most, 2^d a ghost of the GhostFromFiner fill
    const int64_t ghosts =
        std::max({adj_grid(4 * (int64_t)H.src_elem.size(), aops->ghost_block), adj_grid(H.nC, aops->ghost_block),
                  adj_grid((H.nG1 + H.nG2) << c->d, aops->sc_block), adj_grid(H.out_end - H.out_begin, kAdjLinkBlock)});
    interior = std::max({interior, ghosts, (64 * H.nB + block - 1) / block});
    rest = std::max(rest, (64 * H.nBb + block - 1) / block + (H.N - 64 * (H.nB + H.nBb)) / block + 2);
  }
  // the rest of the reverse stream-collide runs beside the interior bricks',
  // so its blocks add to rows of their own
  L.side_row0 = (int)interior;
  L.partial_rows = (int)(interior + rest);
  L.partial = take((size_t)L.partial_rows * kAccCols * 8);
  L.acc = take(32 * 8);
  int64_t max_contrib = 0;
  for (int li = 0; li < c->nlev; ++li) {
    const HostLevel& H = c->M.lv[li];
    const int64_t nsrc = (int64_t)H.src_elem.size();
    L.lam_rec.push_back(take((size_t)nsrc * mom_stride(c->Q) * lb));
    L.recA.push_back(take((size_t)nsrc * mom_stride(c->Q) * lb));
    L.recB.push_back(take((size_t)nsrc * mom_stride(c->Q) * lb));
    L.csr_off.push_back(take((size_t)(nsrc + 1) * 4));
    const int64_t nfine = li + 1 < c->nlev ? c->M.lv[li + 1].nC : 0;
    L.csr_item.push_back(take((size_t)4 * nfine * 4));
    max_contrib = std::max(max_contrib, nfine);
  }
  L.contrib = take((size_t)max_contrib * ((c->Q + 3) / 4 * 4 + 4) * lb);
  for (int li = 0; li < c->nlev; ++li) L.src_saved.push_back(take(c->M.lv[li].src_elem.size() * 4));
  L.state_bytes = align_up((size_t)c->Q * N * c->ops->storage_bytes);
  L.n_ck = (int)((n + K - 1) / K);
  L.n_steps = K;
  L.n_slots = (int)substeps(c, c->n_filled - 1);
  // a step's part of the tape: n_slots states (a state fills only its level's
  // rows of a full-size slot, so the k-th of every level share slot k), then
  // the levels' saves
  L.step_bytes = (size_t)L.n_slots * L.state_bytes;
  for (int li = 0; li < c->nlev; ++li) {
    L.save_off.push_back(L.step_bytes);
    L.save_bytes.push_back(align_up((size_t)c->Q * c->M.lv[li].gsrc_elem.size() * c->ops->storage_bytes));
    if (c->p.time_mode == LBM_TIME_LINEAR && li + 1 < c->nlev) L.step_bytes += L.save_bytes[li] * (size_t)substeps(c, li);
  }
  // workspace rule: record the whole segment when that needs at most twice the
  // states of the step-by-step scheme, or at most 8 GiB
  const size_t by_step = (size_t)K * L.state_bytes + L.step_bytes, whole = (size_t)K * L.step_bytes;
  if (c->p.adjoint_tape == 1) L.tape_all = true;
  else if (c->p.adjoint_tape == 2) L.tape_all = false;
  else L.tape_all = whole <= 2 * by_step || whole <= ((size_t)8 << 30);
  L.ck = o;
  o += (size_t)L.n_ck * L.state_bytes;
  L.steps = o;
  if (!L.tape_all) o += (size_t)L.n_steps * L.state_bytes;
  L.tape = o;
  o += L.step_bytes * (L.tape_all ? (size_t)std::min<int64_t>(K, n) : 1);
  L.fin = o;
  o += L.state_bytes;
  L.total = o;
  return L;
}

// The transposed GhostFromCoarser source lists (ghosts per source, in ghost
// order, then source slot: fixed summation order) and each record's index
// among the sources set aside on the tape.  They depend on the mesh only and
// are built once (0.3 ms a call on the 64^3 two-level mesh).
void build_source_lists(lbm_ctx* c) {
  if (!c->source_lists.empty()) return;
  std::vector<lbm_ctx::SourceLists> all(c->nlev);
  for (int li = 0; li + 1 < c->nlev; ++li) {
    const HostLevel& Hc = c->M.lv[li];
    const HostLevel& Hf = c->M.lv[li + 1];
    lbm_ctx::SourceLists& l = all[li];
    const int64_t nsrc = (int64_t)Hc.src_elem.size();
    l.off.assign(nsrc + 1, 0);
    l.item.resize(4 * Hf.nC);
    for (int64_t k = 0; k < 4 * Hf.nC; ++k) l.off[Hf.gfc_src[k] + 1]++;
    for (int64_t k = 0; k < nsrc; ++k) l.off[k + 1] += l.off[k];
    std::vector<int32_t> fill(l.off.begin(), l.off.end() - 1);
    for (int64_t k = 0; k < Hf.nC; ++k)
      for (int q = 0; q < 4; ++q) l.item[fill[Hf.gfc_src[(size_t)q * Hf.nC + k]]++] = (int32_t)(4 * k + q);
    l.saved.assign(nsrc, -1);
    for (size_t k = 0; k < Hc.gsrc_rec.size(); ++k) l.saved[Hc.gsrc_rec[k]] = (int32_t)k;
  }
  c->source_lists.swap(all);
}

// side stream and fork/join events of the concurrent reverse kernels (ok
// false: not available, everything runs on the bound stream); released when
// the adjoint returns (the driver releases pending resources when done)
struct SideStream {
  cudaStream_t s = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
  bool ok = false;
  SideStream() {
    ok = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&join, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) cudaGetLastError();
  }
  ~SideStream() {
    if (s) cudaStreamDestroy(s);
    if (fork) cudaEventDestroy(fork);
    if (join) cudaEventDestroy(join);
  }
};

}  // namespace

extern "C" {

lbm_status lbm_set_params(lbm_ctx* c, double omega_coarse, const double* u_in) {
  if (!c || !(omega_coarse > 0.0 && omega_coarse < 2.0)) return LBM_ERR_ARG;
  std::vector<double> om(c->nlev);
  om[0] = omega_coarse;
  for (int li = 1; li < c->nlev; ++li) om[li] = finer_omega(om[li - 1], c->p.time_mode);
  for (int li = 0; li < c->nlev; ++li)
    if (std::fabs(1.0 - om[li]) < 1e-3) return c->fail(LBM_ERR_ARG, "omega too close to 1 on some level");
  // the same values again (an optimisation loop over something else) change nothing
  bool same = omega_coarse == c->p.omega_coarse;
  for (int a = 0; u_in && a < 3; ++a) same = same && u_in[a] == c->p.u_in[a];
  if (same) return LBM_OK;
  c->drop_graphs();  // captured steps carry the old omega and inlet values
  c->recs_valid = false;  // the source records depend on omega
  for (int li = 0; li < c->nlev; ++li) c->M.lv[li].omega = om[li];
  c->p.omega_coarse = omega_coarse;
  if (u_in) {
    for (int a = 0; a < 3; ++a) c->p.u_in[a] = u_in[a];
    int cc[kQmax][3];
    double w[kQmax];
    host_lattice(c->Q, cc, w);
    for (int i = 0; i < c->Q; ++i) {
      double cu = 0;
      for (int a = 0; a < c->d; ++a) cu += cc[i][a] * u_in[a];
      c->inlet[i] = 6.0 * w[i] * c->p.rho0 * cu;
    }
  }
  return LBM_OK;
}

lbm_status lbm_adjoint_bytes(lbm_ctx* c, int64_t n_coarse, int32_t K, uint64_t* bytes) {
  if (!c || !bytes || n_coarse < 1 || K < 1) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_adjoint_bytes before lbm_bind");
  if (c->p.time_mode == LBM_TIME_DIFFUSIVE) return c->fail(LBM_ERR_STATE, "no adjoint in LBM_TIME_DIFFUSIVE");
  *bytes = adj_layout(c, n_coarse, K).total;
  return LBM_OK;
}

lbm_status lbm_adjoint(lbm_ctx* c, int64_t n, int32_t K, int32_t objective, void* adj_ws, uint64_t bytes,
                       double* J, double* dJ_dF, double* dJ_domega, double* dJ_duin, double* dJ_df0) {
  if (!c || !adj_ws || n < 1 || K < 1 || objective < 0 || objective > 3) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_adjoint before lbm_bind");
  if (c->p.time_mode == LBM_TIME_DIFFUSIVE) return c->fail(LBM_ERR_STATE, "no adjoint in LBM_TIME_DIFFUSIVE");
  if (objective > c->d) return c->fail(LBM_ERR_ARG, "force component beyond the dimension");
  const AdjLayout L = adj_layout(c, n, K);
  if (bytes < L.total) return c->fail(LBM_ERR_ARG, "adjoint workspace too small");
  if (reinterpret_cast<uintptr_t>(adj_ws) % kAlign) return c->fail(LBM_ERR_ARG, "adjoint workspace not aligned");
  char* W = static_cast<char*>(adj_ws);
  cudaStream_t st = c->st;
  SideStream side, ahead;
  const AdjOps* aops = adj_ops_for(c->p.precision);
  const bool fp64 = c->p.precision == LBM_FP64;
  const size_t N = (size_t)c->M.Ntot;
  auto chk = [&](cudaError_t e, const char* w) { return c->cuda_check(e, w); };
  // ---- clear adjoint state, build the transposed GFC source lists
  lbm_status s = chk(cudaMemsetAsync(W, 0, L.ck, st), "adjoint clear");
  if (s != LBM_OK) return s;
  build_source_lists(c);
  for (int li = 0; li + 1 < c->nlev; ++li) {
    const lbm_ctx::SourceLists& l = c->source_lists[li];
    auto up = [&](size_t to, const std::vector<int32_t>& v) {
      if (s == LBM_OK && !v.empty()) s = chk(cudaMemcpyAsync(W + to, v.data(), v.size() * 4, cudaMemcpyHostToDevice, st), "csr");
    };
    up(L.csr_off[li], l.off);
    up(L.csr_item[li], l.item);
    up(L.src_saved[li], l.saved);
    if (s != LBM_OK) return s;
  }
  auto save_state = [&](char* dst) {
    for (int li = 0; li < c->nlev; ++li) copy_level(c, c->cur(li), dst, li);
  };
  auto restore_state = [&](const char* src, const std::vector<int>& par) {
    c->reset_state_buffers();
    for (int li = 0; li < c->nlev; ++li) {
      c->parity[li] = par[li];
      copy_level(c, src, c->cur(li), li);
    }
    c->recs_valid = false;
  };
  // ---- forward with checkpoints: the parities of every step from a dry walk,
  // then each segment through lbm_step's path (graph replay of step pairs)
  std::vector<std::vector<int>> parity_at(n + 1);
  {
    const std::vector<int> p0 = c->parity;
    c->dry = true;
    for (int64_t t = 0; t < n; ++t) {
      parity_at[t] = c->parity;
      c->advance(0);
    }
    c->dry = false;
    parity_at[n] = c->parity;
    c->parity = p0;
  }
  // however this call ends, the context is back on its own two buffers
  struct Buffers {
    lbm_ctx* c;
    ~Buffers() {
      c->new_state = nullptr;
      c->at_mid_step = nullptr;
      c->reset_state_buffers();
    }
  } buffers{c};
  // rows [at, at + cnt) of level li
  auto copy_rows_of = [&](const void* from, void* to, int li, int64_t at, int64_t cnt) {
    const size_t sb = c->ops->storage_bytes;
    launch_copy_rows(from, to, N * sb, (size_t)(c->M.lv[li].base + at) * sb, (size_t)cnt * sb, c->Q, sb, st);
  };
  // runs one coarse step, its new states going to the tape's part at `part`
  auto record_step = [&](Recorded& r, char* part) {
    r.states.assign(c->nlev, {});
    r.mids.assign(c->nlev, {});
    c->ensure_records();
    for (int li = 0; li < c->nlev; ++li) r.states[li].push_back(c->cur(li));
    c->new_state = [&](int li) -> void* {
      char* slot = part + (r.states[li].size() - 1) * L.state_bytes;
      r.states[li].push_back(slot);
      // slots that no op of the step writes before they are read: an outer
      // GhostFromFiner ghost that is a source, at t + 1 (no mesh has one so far)
      if (c->ld[li].n_gsrc > c->ld[li].n_gsrc_inner) copy_rows_of(c->nxt(li), slot, li, c->M.lv[li].oG2, c->M.lv[li].nG2);
      return slot;
    };
    c->at_mid_step = [&](int li) {
      const HostLevel& H = c->M.lv[li];
      char* to = part + L.save_off[li] + r.mids[li].size() * L.save_bytes[li];
      r.mids[li].push_back(to);
      launch_gather_elements(c->cur(li), to, c->at<int32_t>(c->ld[li].gsrc_elem), (int64_t)H.gsrc_elem.size(), (int64_t)N,
                             c->Q, c->ops->storage_bytes, st);
    };
    if (c->timing != 1 && c->can_batch()) c->step_batched();
    else c->advance(0);
    c->new_state = nullptr;
    c->at_mid_step = nullptr;
  };
  std::vector<Recorded> recs(L.tape_all ? std::min<int64_t>(K, n) : 1);
  for (int64_t t = 0; t < n && s == LBM_OK; t += K) {
    if (L.tape_all && t + K >= n) {
      // the last segment is recorded as the forward passes through it
      for (int64_t k = t; k < n; ++k) record_step(recs[k - t], W + L.tape + (size_t)(k - t) * L.step_bytes);
      s = c->launched("adjoint forward");
    } else {
      save_state(W + L.ck + (size_t)(t / K) * L.state_bytes);
      s = c->run_steps(std::min<int64_t>(K, n - t));
    }
  }
  if (s == LBM_OK && c->parity != parity_at[n]) s = c->fail(LBM_ERR_INTERNAL, "adjoint forward parities differ");
  if (s != LBM_OK) return s;
  save_state(W + L.fin);
  if (L.tape_all) {
    // The ghost slots that no stream-collide writes, as lbm_step leaves them:
    // what the fills put into the same buffer two substeps earlier, and in
    // LINEAR mode the outer GhostFromCoarser layer, which the steps leave
    // alone, as the context's buffer holds it.
    const bool linear = c->p.time_mode == LBM_TIME_LINEAR;
    for (int li = 0; li < c->nlev; ++li) {
      const HostLevel& H = c->M.lv[li];
      std::vector<const void*> seq;  // the states of the recorded steps
      for (int64_t k = 0; k < n - (int64_t)(L.n_ck - 1) * K; ++k)
        seq.insert(seq.end(), recs[k].states[li].begin() + (k ? 1 : 0), recs[k].states[li].end());
      const void* own = parity_at[n][li] ? c->at(c->oB) : c->at(c->oA);
      const void* before = seq.size() >= 3 ? seq[seq.size() - 3] : own;
      if (linear) {
        launch_copy_ghosts(before, own, W + L.fin, c->at<uint8_t>(c->ld[li].gfc_oct), H.base + H.oC, H.nC, (int64_t)N, c->Q,
                           c->ops->storage_bytes, st);
        copy_rows_of(before, W + L.fin, li, H.oG2, H.nG2);
      } else {
        copy_rows_of(before, W + L.fin, li, H.oG1, H.nG1);
        copy_rows_of(before, W + L.fin, li, H.oG2, H.nG2);
      }
    }
  }
  s = c->launched("adjoint forward");
  if (s != LBM_OK) return s;
  // ---- objective and seed
  double red[8];
  s = lbm_reduce(c, red);
  if (s != LBM_OK) return s;
  if (J) *J = objective == 0 ? red[7] : red[3 + objective];
  char* lamA = W + L.lamA;
  char* lamB = W + L.lamB;
  auto lam_for = [&](int par) { return par ? lamB : lamA; };
  // the body-force adjoint is accumulated only when it is asked for
  double* lamF = dJ_dF ? reinterpret_cast<double*>(W + L.lamF) : nullptr;
  double* partial = reinterpret_cast<double*>(W + L.partial);
  double* acc = reinterpret_cast<double*>(W + L.acc);
  const void* force = c->force_ptr();
  auto common = [&](const void* fsrc, void* la, void* lbuf, int acc_la = 0, int acc_lb = -1) {
    AdjCommon cm{};
    cm.la = acc_la;
    cm.lb = acc_lb;
    cm.fsrc = fsrc;
    cm.force = force;
    cm.lam_a = la;
    cm.lam_b = lbuf;
    cm.lam_force = lamF;
    cm.partial = partial;
    cm.Ntot = (int64_t)N;
    cm.rho_off = c->rho_off;
    cm.rho0 = c->p.rho0;
    return cm;
  };
  for (int li = 0; li < c->nlev; ++li) {
    const HostLevel& H = c->M.lv[li];
    AdjSeedArgs a{};
    a.c = common(c->cur(li), nullptr, lam_for(c->parity[li]));
    a.objective = objective;
    a.begin = H.base + H.oF;
    a.end = H.base + H.oF + H.nF;
    a.vol = std::ldexp(1.0, -c->d * li);
    a.obs_elem = c->at<int32_t>(c->oObsElem) + H.obs_begin;
    a.obs_dir = c->at<int8_t>(c->oObsDir) + H.obs_begin;
    a.obs_a = c->at<int32_t>(c->oObsA) + H.obs_begin;
    a.obs_q = c->at<double>(c->oObsQ) + H.obs_begin;
    a.obs_n = H.obs_end - H.obs_begin;
    a.fscale = std::ldexp(1.0, (c->d - 1) * (c->nlev - 1 - li));
    if (objective == 0) {
      if (a.end > a.begin) aops->seed(c->Q, a, st);
    } else if (a.obs_n > 0) {
      // the own slot, then (interpolated bounce-back only) the second node and
      // the opposite slot, one pass each so that no two links share a slot
      for (int which = 0; which < (c->p.bouzidi ? 3 : 1); ++which) {
        a.which = which;
        aops->seed(c->Q, a, st);
      }
    }
  }
  // ---- reverse sweep
  const int nseg = L.n_ck;
  // the op sequence depends only on the starting parity of the coarsest level
  std::vector<TapeOp> plans[2];
  auto plan = [&](const std::vector<int>& par) -> const std::vector<TapeOp>& {
    std::vector<TapeOp>& t = plans[par[0] & 1];
    if (t.empty()) {
      const std::vector<int> p0 = c->parity;
      c->parity = par;
      t = plan_step(c);
      c->parity = p0;
    }
    return t;
  };
  // runs one recorded step backwards
  auto reverse_step = [&](const Recorded& r, const std::vector<TapeOp>& tape) {
    auto saved = [&](int li, int mid) {
      return SavedSources{r.mid(li, mid), reinterpret_cast<const int32_t*>(W + L.src_saved[li]),
                          (int64_t)c->M.lv[li].gsrc_elem.size()};
    };
    // forward records of an interface from the tape's states: at t, and for
    // the fill at t + 1/2 (kb >= 0) the means of those at t and t + 1
    auto records = [&](int lc, int ka, int kb, int mid, cudaStream_t st) {
      const HostLevel& Hc = c->M.lv[lc];
      MomentsArgs m{};
      m.force = force;
      m.elem = c->at<int32_t>(c->ld[lc].src_elem);
      m.Ntot = (int64_t)N;
      m.nsrc = c->ld[lc].nsrc;
      m.rx = make_relax(c->Q, Hc.omega);
      m.rx32 = make_relax32(Hc.omega);
      m.rho_off = c->rho_off;
      m.rho_off32 = (float)c->rho_off;
      m.src = r.state(lc, ka);
      m.mom = W + L.recA[lc];
      // LINEAR mode reverses the fill at t + 1/2 first, which has formed these
      if (kb >= 0 || c->p.time_mode != LBM_TIME_LINEAR) c->ops->source_moments(c->Q, m, st);
      if (kb < 0) return static_cast<const void*>(W + L.recA[lc]);
      m.src = r.state(lc, kb);
      m.saved = saved(lc, mid);
      m.mom = W + L.recB[lc];
      m.prev = W + L.recA[lc];
      c->ops->source_moments(c->Q, m, st);
      return static_cast<const void*>(W + L.recB[lc]);
    };
    const void* ready = nullptr;  // records formed ahead of the fill whose reverse comes next
    for (int k = (int)tape.size() - 1; k >= 0; --k) {
      const TapeOp& t = tape[k];
      const int li = t.level;
      const HostLevel& H = c->M.lv[li];
      if (t.op == OP_SC) {
        const int p = t.parity[li];
        const bool outlet = H.out_end > H.out_begin;
        if (outlet) {
          OutletArgs o = c->outlet_args(W + L.side_fwd);
          c->add_outlet(o, li, r.state(li, t.k));
          c->ops->outlet(c->Q, o, st);
        }
        AdjSCArgs a{};
        a.c = common(r.state(li, t.k), lam_for(!p), lam_for(p), li);
        a.nbr = c->at<uint32_t>(c->oNbr);
        a.side_fwd = W + L.side_fwd;
        a.lam_side = W + L.lam_side;
        a.omega = H.omega;
        std::memcpy(a.inlet, c->inlet, sizeof(a.inlet));
        a.inlet_s = c->at<double>(c->oInletS);
        // bricks through the brick tables, the rest through the neighbour
        // list, beside the interior bricks on the side stream
        const int64_t nbrick = 64 * (H.nB + H.nBb);
        a.begin = H.base + H.oF;
        a.n_interior = H.nB;
        a.n_boundary = H.nBb;
        a.brick_nb = c->at<int32_t>(c->oBrickNb) + (size_t)H.brick_first * 27;
        a.brick_tab = c->at<uint16_t>(c->oBrickTab);
        if (c->p.time_mode == LBM_TIME_TWO_LAYER) {
          a.list_begin = H.base + H.oC;
          a.list_end = H.base + H.oG1 - nbrick;
          a.hole_at = H.base + H.oF;
          a.hole_len = nbrick;
        } else {
          a.list_begin = H.base + H.oF + nbrick;
          a.list_end = H.base + H.oG2;
          a.hole_at = a.list_end;
          a.hole_len = 0;
        }
        a.row0 = L.side_row0;
        // beside both, the records that the reverse of this level's ghost fill
        // reads next (they depend on the tape only)
        if (k > 0 && ahead.ok) {
          const int f = k - 1;
          if ((tape[f].op == OP_GFC_A || tape[f].op == OP_GFC_B) && c->M.lv[tape[f].level].nC > 0) {
            cudaEventRecord(ahead.fork, st);
            cudaStreamWaitEvent(ahead.s, ahead.fork, 0);
            ready = records(tape[f].level - 1, tape[f].k, tape[f].op == OP_GFC_B ? tape[f].kb : -1, tape[f].mid, ahead.s);
            cudaEventRecord(ahead.join, ahead.s);
          }
        }
        const bool fork = side.ok && H.nB > 0;
        if (fork) {
          cudaEventRecord(side.fork, st);
          cudaStreamWaitEvent(side.s, side.fork, 0);
        }
        aops->sc_interior(c->Q, a, st);
        aops->sc_rest(c->Q, a, fork ? side.s : st);
        if (fork) {
          cudaEventRecord(side.join, side.s);
          cudaStreamWaitEvent(st, side.join, 0);
        }
        if (outlet) {
          for (int which = 0; which < (c->p.bouzidi ? 6 : 3); ++which) {
            AdjOutletArgs o{};
            o.c = common(r.state(li, t.k), nullptr, lam_for(p), li);
            o.elem = c->at<int32_t>(c->oOutElem);
            o.a = c->at<int32_t>(c->oOutA);
            o.b = c->at<int32_t>(c->oOutB);
            o.dir = c->at<int8_t>(c->oOutDir);
            o.kind = c->at<int8_t>(c->oOutKind);
            o.lam_side = W + L.lam_side;
            o.begin = H.out_begin;
            o.end = H.out_end;
            o.which = which;
            o.omega = H.omega;
            o.zero_gradient = c->p.outlet == LBM_OUTLET_ZERO_GRADIENT;
            o.q = c->at<double>(c->oOutQ);
            aops->outlet(c->Q, o, st);  // pass 0 also adds d/d omega through the normal links' f^neq
          }
        }
      } else if (t.op == OP_MOM_A || t.op == OP_MOM_B) {
        if (c->ld[li].nsrc == 0) continue;
        // the fill of the finer level's ghosts has just been reversed into contrib
        const bool half = t.op == OP_MOM_B;
        AdjMomArgs a{};
        a.c = common(r.state(li, t.k), nullptr, lam_for(t.parity[li]), li);
        a.elem = c->at<int32_t>(c->ld[li].src_elem);
        if (half) a.saved = saved(li, t.mid);
        a.contrib = W + L.contrib;
        a.off = reinterpret_cast<const int32_t*>(W + L.csr_off[li]);
        a.item = reinterpret_cast<const int32_t*>(W + L.csr_item[li]);
        a.rec_half = c->p.time_mode == LBM_TIME_LINEAR ? W + L.lam_rec[li] : nullptr;
        a.half = half;
        a.nsrc = c->ld[li].nsrc;
        a.omega = H.omega;
        aops->moments(c->Q, a, st);
      } else if (t.op == OP_GFC_A || t.op == OP_GFC_B) {
        if (H.nC == 0) continue;
        const int lc = li - 1;
        if (ready) cudaStreamWaitEvent(st, ahead.join, 0);
        const void* rec = ready ? ready : records(lc, t.k, t.op == OP_GFC_B ? t.kb : -1, t.mid, st);
        ready = nullptr;
        AdjGfcArgs a{};
        a.c = common(nullptr, lam_for(t.parity[li]), nullptr, lc, li);
        a.rec = rec;
        a.gsrc = c->at<int32_t>(c->ld[li].gfc_src);
        a.oct = c->at<uint8_t>(c->ld[li].gfc_oct);
        a.contrib = W + L.contrib;
        a.ng = H.nC;
        a.dest0 = H.base + H.oC;
        a.omega_c = c->M.lv[lc].omega;
        a.omega_f = H.omega;
        aops->gfc(c->Q, a, st);
      } else if (t.op == OP_GFF) {
        if (H.nG1 + H.nG2 == 0) continue;
        AdjGffArgs a{};
        a.c = common(r.state(li + 1, t.k), lam_for(t.parity[li]), lam_for(t.parity[li + 1]), li, li + 1);
        a.child0 = c->at<int32_t>(c->ld[li].gff_child0);
        a.ng = H.nG1 + H.nG2;
        a.n_inner = H.nG1;
        a.dest0 = H.base + H.oG1;
        a.dest_outer = H.base + H.oG2;
        a.omega_c = H.omega;
        a.omega_f = c->M.lv[li + 1].omega;
        aops->gff(c->Q, a, st);
      }
    }
    return c->launched("adjoint sweep");
  };
  for (int seg = nseg - 1; seg >= 0 && s == LBM_OK; --seg) {
    const int64_t s0 = (int64_t)seg * K, s1 = std::min<int64_t>(s0 + K, n);
    if (L.tape_all) {
      if (s1 < n) {
        restore_state(W + L.ck + (size_t)seg * L.state_bytes, parity_at[s0]);
        for (int64_t t = s0; t < s1; ++t) record_step(recs[t - s0], W + L.tape + (size_t)(t - s0) * L.step_bytes);
      }
      for (int64_t t = s1 - 1; t >= s0 && s == LBM_OK; --t) s = reverse_step(recs[t - s0], plan(parity_at[t]));
    } else {
      // recompute the segment keeping each step's start state; the last step's
      // is the live state, which its recording starts from directly
      restore_state(W + L.ck + (size_t)seg * L.state_bytes, parity_at[s0]);
      for (int64_t t = s0; t + 1 < s1 && s == LBM_OK; ++t) {
        save_state(W + L.steps + (size_t)(t - s0) * L.state_bytes);
        s = c->run_steps(1);
      }
      for (int64_t t = s1 - 1; t >= s0 && s == LBM_OK; --t) {
        if (t + 1 < s1) restore_state(W + L.steps + (size_t)(t - s0) * L.state_bytes, parity_at[t]);
        record_step(recs[0], W + L.tape);
        s = reverse_step(recs[0], plan(parity_at[t]));
      }
    }
  }
  if (s != LBM_OK) return s;
  // ---- parameter gradients
  launch_accum(AccumArgs{partial, L.partial_rows, acc}, st);
  double hacc[kAccCols];
  s = chk(cudaMemcpyAsync(hacc, acc, sizeof(hacc), cudaMemcpyDeviceToHost, st), "adjoint acc");
  if (s == LBM_OK) s = chk(cudaStreamSynchronize(st), "adjoint sync");
  if (s != LBM_OK) return s;
  if (dJ_domega) {
    // omega_L = 1 / (1/2 + 2^L (1/omega_c - 1/2)): d omega_L / d omega_c = 2^L omega_L^2 / omega_c^2
    const double wc = c->M.lv[0].omega;
    double g = 0.0;
    for (int li = 0; li < c->nlev; ++li) {
      const double wl = c->M.lv[li].omega;
      g += hacc[li] * std::ldexp(1.0, li) * wl * wl / (wc * wc);
    }
    *dJ_domega = g;
  }
  if (dJ_duin)
    for (int a = 0; a < 3; ++a) dJ_duin[a] = a < c->d ? hacc[16 + a] : 0.0;
  if (dJ_dF) {
    double* stage = c->at<double>(c->oStage);
    for (int64_t first = 0; first < c->M.n_user; first += c->chunk) {
      const int64_t cnt = std::min<int64_t>(c->chunk, c->M.n_user - first);
      launch_gather_force_user(lamF, c->at<int32_t>(c->oUslot), stage, first, cnt, (int64_t)N, c->d, st);
      s = chk(cudaMemcpyAsync(dJ_dF + first * c->d, stage, cnt * c->d * 8, cudaMemcpyDeviceToHost, st), "dJdF");
      if (s == LBM_OK) s = chk(cudaStreamSynchronize(st), "dJdF sync");
      if (s != LBM_OK) return s;
    }
  }
  if (dJ_df0) {
    // the adjoint now holds dJ / d(initial pdfs), in the buffers of the parities at t0
    uint32_t pm = 0;
    for (int li = 0; li < c->nlev; ++li) pm |= (uint32_t)(parity_at[0][li] & 1) << li;
    double* stage = c->at<double>(c->oStage);
    for (int64_t first = 0; first < c->M.n_user; first += c->chunk) {
      const int64_t cnt = std::min<int64_t>(c->chunk, c->M.n_user - first);
      launch_gather_lam_user(fp64, lamA, lamB, pm, c->at<int32_t>(c->oUslot), c->at<uint8_t>(c->oUlev), stage,
                             first, cnt, (int64_t)N, c->Q, st);
      s = chk(cudaMemcpyAsync(dJ_df0 + first * c->Q, stage, cnt * c->Q * 8, cudaMemcpyDeviceToHost, st), "dJdf0");
      if (s == LBM_OK) s = chk(cudaStreamSynchronize(st), "dJdf0 sync");
      if (s != LBM_OK) return s;
    }
  }
  // ---- leave the simulation at the final state
  restore_state(W + L.fin, parity_at[n]);
  s = c->launched("adjoint restore");
  if (s == LBM_OK) s = chk(cudaStreamSynchronize(st), "adjoint end");
  return s;
}

}  // extern "C"
