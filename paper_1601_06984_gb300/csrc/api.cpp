// C ABI of liblbm (include/lbm.h): context, device workspace layout, the
// recursive level time stepping driver (Sec. 2.2) and the host<->device
// transfers of the public calls.
#include <cuda_runtime_api.h>

#include <unistd.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "lbm_ctx.h"
#include "lbm_internal.h"

using namespace lbm;

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }


}  // namespace

using lbm::LevelDev;

void lbm_ctx::layout() {
  const HostMesh& m = M;
  size_t o = 0;
  auto take = [&](size_t b) {
    size_t r = o;
    o += align_up(std::max<size_t>(b, 1));
    return r;
  };
  const size_t sb = ops->storage_bytes, cb = ops->compute_bytes;
  const size_t N = (size_t)m.Ntot;
  oA = take(Q * N * sb);
  oB = take(Q * N * sb);
  oNbr = take((size_t)(Q - 1) * N * 4);
  oBrickNb = take(m.brick_nb.size() * 4);
  oBrickTab = take(m.brick_tab.size() * 2);
  oInletS = take(m.inlet_s.size() * 8);
  oOutQ = take(m.out_q.size() * 8);
  oObsA = take(m.obs_a.size() * 4);
  oObsQ = take(m.obs_q.size() * 8);
  oF = p.use_force ? take((size_t)d * N * cb) : 0;
  ld.assign(nlev, LevelDev());
  const size_t M_ = mom_stride(Q);
  for (int li = 0; li < nlev; ++li) {
    const HostLevel& H = m.lv[li];
    LevelDev& L = ld[li];
    L.gff_child0 = take(H.gff_child0.size() * 4);
    L.gfc_src = take(H.gfc_src.size() * 4);
    L.gfc_oct = take(H.gfc_oct.size());
    L.src_elem = take(H.src_elem.size() * 4);
    L.nsrc = (int64_t)H.src_elem.size();
    L.gsrc_elem = take(H.gsrc_elem.size() * 4);
    L.gsrc_rec = take(H.gsrc_rec.size() * 4);
    L.n_gsrc = (int64_t)H.gsrc_elem.size();
    L.n_gsrc_inner = H.n_gsrc_inner;
    L.momA[0] = take(M_ * L.nsrc * cb);
    L.momA[1] = take(M_ * L.nsrc * cb);
  }
  const size_t nout = m.out_elem.size(), nobs = m.obs_elem.size();
  oOutElem = take(nout * 4);
  oOutA = take(nout * 4);
  oOutB = take(nout * 4);
  oOutDir = take(nout);
  oOutKind = take(nout);
  oSide = take(nout * cb);
  oObsElem = take(nobs * 4);
  oObsDir = take(nobs);
  oUslot = take((size_t)m.n_user * 4);
  oUlev = take((size_t)m.n_user);
  oSlotUser = take((size_t)N * 4);
  oSrcMask = take(m.src_mask.size() * 4);
  oSrcFirst = take(m.src_first.size() * 4);
  chunk = std::min<int64_t>(m.n_user, (int64_t)1 << 20);
  oStage = take((size_t)chunk * (1 + d + nS + Q + Q) * 8);
  oPartial = take((size_t)nlev * kReduceBlocks * 8 * 8);
  oRed = take(8 * 8);
  bytes = o;
  n_filled = 1;
  for (int li = 0; li < nlev; ++li)
    if (m.lv[li].nF > 0) n_filled = li + 1;
  outlet_reads_ghosts = false;
  for (const auto* v : {&m.out_elem, &m.out_a, &m.out_b})
    for (int32_t e : *v)
      if (e >= 0 && m.kind[e] != K_FLUID) outlet_reads_ghosts = true;
}

// ---------------------------------------------------------------- driver
// unit conversion into the ghosts' level: fine -> coarse u_c = (dt_c / dt_f) / 2
// u_f, the density deviation with the square of that factor (1 in acoustic
// scaling); coarse -> fine the inverse
template <class Args>
void lbm_ctx::ghost_units(Args& a, bool to_coarse) const {
  const double m = time_ratio(p.time_mode), us = to_coarse ? m / 2.0 : 2.0 / m;
  const double odd = odd_fneq_ratio(p.time_mode, to_coarse), rs = us * us, shift = (1.0 - rs) * (p.rho0 - rho_off);
  a.u64 = {rho_off, m, us, rs, shift, odd};
  a.u32 = {(float)rho_off, (float)m, (float)us, (float)rs, (float)shift, (float)odd};
  a.odd_rescale = odd != 1.0;
  a.Ntot = M.Ntot;
}

GffArgs lbm_ctx::gff_args() const {
  GffArgs a{};
  ghost_units(a, true);
  a.force = force_ptr();
  a.sources = source_table();
  return a;
}

void lbm_ctx::add_gff(GffArgs& a, int li) const {
  const HostLevel& H = M.lv[li];
  const HostLevel& Hf = M.lv[li + 1];
  if (H.nG1 + H.nG2 == 0) return;
  const int k = a.nseg++;
  GffLevel& L = a.lev[k];
  L.src_fine = cur(li + 1);
  L.child0 = at<int32_t>(ld[li].gff_child0);
  L.ng = (int32_t)(H.nG1 + H.nG2);
  L.n_inner = (int32_t)H.nG1;
  L.dest0 = (int32_t)(H.base + H.oG1);
  L.dest_outer = (int32_t)(H.base + H.oG2);
  L.dst = cur(li);
  L.rec_out = ld[li].n_gsrc > 0 ? at(ld[li].momA[parity[li]]) : nullptr;
  L.rx_f = make_relax32(Hf.omega);
  a.rx_c[k] = make_relax32(H.omega);
  a.rx_c64[k] = make_relax(Q, H.omega);
  a.rx_f64[k] = make_relax(Q, Hf.omega);
  const double m = time_ratio(p.time_mode);
  a.scale[k] = (1.0 - H.omega) * m * Hf.omega / H.omega / (1 << d);
  const float wc = (float)H.omega, wf = (float)Hf.omega;  // the FP32 kernels' factor, in their arithmetic
  L.scale32 = (1.0f - wc) * (float)m * wf / wc * (1.0f / (float)(1 << d));
}

void lbm_ctx::fill_gff(int li) {
  GffArgs a = gff_args();
  add_gff(a, li);
  if (!a.nseg) return;
  timed_launch(li, TK_GFF, [&] { issued += ops->fill_gff(Q, a, st); });
  ++launches;
}

SourceTable lbm_ctx::source_table() const { return {at<uint32_t>(oSrcMask), at<int32_t>(oSrcFirst)}; }

void lbm_ctx::source_moments(int li, size_t mom_off, cudaStream_t s, int subset) {
  const LevelDev& L = ld[li];
  const int64_t n = subset == SRC_ALL ? L.nsrc : L.n_gsrc - L.n_gsrc_inner;
  if (n == 0) return;
  if (!s) s = st;
  MomentsArgs a{};
  a.src = cur(li);
  a.force = force_ptr();
  if (subset == SRC_ALL) {
    a.elem = at<int32_t>(L.src_elem);
  } else {
    a.elem = at<int32_t>(L.gsrc_elem) + L.n_gsrc_inner;
    a.rec = at<int32_t>(L.gsrc_rec) + L.n_gsrc_inner;
  }
  a.mom = at(mom_off);
  a.Ntot = M.Ntot;
  a.nsrc = n;
  a.rx = make_relax(Q, M.lv[li].omega);
  a.rx32 = make_relax32(M.lv[li].omega);
  a.rho_off = rho_off;
  a.rho_off32 = (float)rho_off;
  timed_launch(li, TK_MOM, [&] { issued += ops->source_moments(Q, a, s); }, s);
  ++launches;
}

GfcArgs lbm_ctx::gfc_args() const {
  GfcArgs a{};
  ghost_units(a, false);
  return a;
}

void lbm_ctx::add_gfc(GfcArgs& a, int lf, bool two_times, bool all_layers) const {
  const HostLevel& H = M.lv[lf];
  if (H.nC == 0) return;
  const int lc = lf - 1;
  GfcLevel& L = a.lev[a.nseg++];
  // at t + 1/2 (after the coarse stream-collide): the means of the records
  // at t and t + 1, which the two buffers hold
  L.mom = at(ld[lc].momA[parity[lc] ^ (two_times ? 1 : 0)]);
  L.mom2 = two_times ? at(ld[lc].momA[parity[lc]]) : nullptr;
  L.gsrc = at<int32_t>(ld[lf].gfc_src);
  L.oct = at<uint8_t>(ld[lf].gfc_oct);
  L.ng = (int32_t)H.nC;
  L.dest0 = (int32_t)(H.base + H.oC);
  L.dst = cur(lf);
  L.skip_outer = !all_layers && p.time_mode == LBM_TIME_LINEAR;
  const double wc = M.lv[lc].omega, wf = H.omega, m = time_ratio(p.time_mode);
  L.scale = (1.0 - wf) * wc / (m * wf);
  const float wcf = (float)wc, wff = (float)wf;  // the FP32 kernels' factor, in their arithmetic
  L.scale32 = (1.0f - wff) * wcf / ((float)m * wff);
}

void lbm_ctx::fill_gfc(int lf, bool two_times, bool all_layers) {
  GfcArgs a = gfc_args();
  add_gfc(a, lf, two_times, all_layers);
  if (!a.nseg) return;
  timed_launch(lf, TK_GFC, [&] { issued += ops->fill_gfc(Q, a, st); });
  ++launches;
}

OutletArgs lbm_ctx::outlet_args(const void* side) const {
  OutletArgs o{};
  o.side = const_cast<void*>(side);
  o.elem = at<int32_t>(oOutElem);
  o.a = at<int32_t>(oOutA);
  o.b = at<int32_t>(oOutB);
  o.dir = at<int8_t>(oOutDir);
  o.kind = at<int8_t>(oOutKind);
  o.force = force_ptr();
  o.Ntot = M.Ntot;
  o.rho_off = rho_off;
  o.rho0 = p.rho0;
  o.zero_gradient = p.outlet == LBM_OUTLET_ZERO_GRADIENT;
  o.q = at<double>(oOutQ);
  return o;
}

void lbm_ctx::add_outlet(OutletArgs& o, int li, const void* src) const {
  const HostLevel& H = M.lv[li];
  if (H.out_end == H.out_begin) return;
  if (!o.nlev) o.begin = H.out_begin;  // consecutive levels' links are consecutive
  OutletLevel& L = o.lev[o.nlev++];
  L.src = src;
  L.end = H.out_end;
  L.omega = H.omega;
}

ScArgs lbm_ctx::sc_args() const {
  ScArgs a{};
  a.force = force_ptr();
  a.tab = at<uint16_t>(oBrickTab);
  a.nbr = at<uint32_t>(oNbr);
  a.side = at(oSide);
  a.inlet_s = at<double>(oInletS);
  a.sources = source_table();
  a.Ntot = M.Ntot;
  a.rho_off = rho_off;
  a.rho_off32 = (float)rho_off;
  for (int i = 0; i < kQmax; ++i) a.inlet[i] = inlet[i];
  return a;
}

int lbm_ctx::add_sc(ScArgs& a, int slot, int li, int kind) const {
  const HostLevel& H = M.lv[li];
  // interior bricks, then boundary bricks are the first 64 (nB + nBb) fluid
  // elements; the rest goes through the neighbour list: TWO_LAYER and
  // DIFFUSIVE [GFC | fluid], LINEAR [fluid | GFF inner], minus the bricks
  const int64_t nbrick = 64 * (H.nB + H.nBb);
  ScSeg g{};
  g.nb = at<int32_t>(oBrickNb) + (size_t)H.brick_first * 27;
  int64_t begin = H.base + H.oF, n = 0;
  if (kind == TK_INTERIOR) {
    n = H.nB;
  } else if (kind == TK_BOUNDARY) {
    g.nb += (size_t)H.nB * 27;
    begin += 64 * H.nB;
    n = H.nBb;
  } else {
    g.list = 1;
    if (p.time_mode != LBM_TIME_LINEAR) {
      g.hole_at = (int32_t)begin;
      g.hole_len = (int32_t)nbrick;
      begin = H.base + H.oC;
      n = H.base + H.oG1 - nbrick - begin;
    } else {
      begin += nbrick;
      n = H.base + H.oG2 - begin;
      g.hole_at = (int32_t)(begin + n);
    }
  }
  if (n <= 0) return 0;
  g.begin = (int32_t)begin;
  g.n = (int32_t)n;
  g.src = cur(li);
  g.dst = nxt(li);
  g.rx = make_relax32(H.omega);
  g.uin = (float)level_velocity_ratio(li, p.time_mode);  // a power of two
  // the level's GFC source records at t + 1 from the new state
  if (li + 1 < nlev && ld[li].nsrc > 0) g.rec_out = at(ld[li].momA[parity[li] ^ 1]);
  g.level = (int16_t)slot;
  a.rx[slot] = make_relax(Q, H.omega);
  a.seg[a.nseg++] = g;
  return 1;
}

void lbm_ctx::stream_collide(int li) {
  if (new_state) state[li][parity[li] ^ 1] = new_state(li);
  OutletArgs o = outlet_args(at(oSide));
  add_outlet(o, li, cur(li));
  if (o.nlev) {
    timed_launch(li, TK_OUTLET, [&] { issued += ops->outlet(Q, o, st); });
    ++launches;
  }
  for (int kind : {TK_INTERIOR, TK_BOUNDARY, TK_LIST}) {
    ScArgs a = sc_args();
    if (!add_sc(a, 0, li, kind)) continue;
    timed_launch(li, kind, [&] { issued += (kind == TK_INTERIOR ? ops->sc_interior : ops->sc_rest)(Q, p.use_force != 0, a, st); });
    ++launches;
  }
  parity[li] ^= 1;
}

// One coarse step, all levels that advance at the same instant together.
// With r the time-step ratio and T = r^(n-1) ticks of the finest level in a
// coarse step, level l advances at the ticks that are multiples of
// r^(n-1-l); the levels advancing at a tick are l0..n-1.  At such an instant
// the order the recursion (advance()) gives them is not needed: a
// GhostFromFiner ghost reads fluid children only, a GhostFromCoarser ghost
// the records of fluid and GhostFromFiner sources only, and a level's
// stream-collide its own state, so three launches serve all levels:
//   the GhostFromFiner fills of l0..n-2 with their ghosts' records,
//   the GhostFromCoarser fills of l0+1..n-1 (and, in LINEAR mode, that of l0
//   at the middle of the coarser level's step),
//   the stream-collide of l0..n-1 (interior bricks beside the rest).
// The four-level cylinder has 20 such launches in a row instead of 36, the
// five-level sphere 40 instead of 76, two-level flows 5 instead of 7, and
// small levels share a launch (cylinder 109 -> 67 us a coarse step, 56 us
// with the launches chained; sphere of 1.1e7 elements 5.08 -> 4.94 ms).
// Every op has the inputs it has in advance(): same results bit for bit.
// Starting the interior bricks, which read no ghost, beside the GhostFromFiner
// fill slowed both (two-level 64^3, FP32: 50 against 48 us; FP64 D2Q9: 84
// against 40 us), and taking them into the other stream-collide launch cost
// more than the fork it saves (49 against 48 us).
void lbm_ctx::step_batched() {
  const int n = n_filled, r = time_ratio(p.time_mode);
  int64_t T = 1;
  for (int l = 1; l < n; ++l) T *= r;
  for (int64_t tick = 0; tick < T; ++tick) {
    int l0 = n - 1;
    for (int64_t period = r; l0 > 0 && tick % period == 0; period *= r) --l0;
    tick_batched(l0, n);
  }
  // levels declared beyond the finest one present hold no element; each takes
  // an even number of substeps per coarse step
}

void lbm_ctx::tick_batched(int l0, int n) {
  const bool finest_only = l0 == n - 1;
  const int timed_level = finest_only ? n - 1 : -1;
  auto fork = [&](int b) {
    cudaEventRecord(br.fork[b], st);
    cudaStreamWaitEvent(br.s[b], br.fork[b], 0);
  };
  auto join = [&](int b) {
    cudaEventRecord(br.join[b], br.s[b]);
    cudaStreamWaitEvent(st, br.join[b], 0);
  };
  if (new_state)
    for (int l = l0; l < n; ++l) state[l][parity[l] ^ 1] = new_state(l);
  ScArgs in = sc_args(), rest = sc_args(), rest_fin = sc_args();
  OutletArgs out = outlet_args(at(oSide));
  int64_t elements = 0;
  for (int l = l0; l < n; ++l) elements += M.lv[l].nF;
  const bool beside = elements <= kBesideElements;
  for (int l = l0; l < n; ++l) {
    // large instants: the finest level's rest apart, without record epilogue
    ScArgs& r = beside || finest_only || l + 1 < n ? rest : rest_fin;
    launches += add_sc(in, l - l0, l, TK_INTERIOR);
    launches += add_sc(r, l - l0, l, TK_BOUNDARY);
    launches += add_sc(r, l - l0, l, TK_LIST);
    const int no = out.nlev;
    add_outlet(out, l, cur(l));
    launches += out.nlev - no;
  }
  const bool chain = capturing && elements <= (p.precision == LBM_FP64 ? kChainElements64 : kChainElements);
  rest.chain = chain;
  const bool force = p.use_force != 0;
  // Interior bricks read no ghost.  At small instants they run beside the
  // GhostFromCoarser fill; beyond kBesideElements only after it: the fill
  // leaves an SM little L1 beside its shared memory, bricks that start there
  // keep that split for as long as blocks follow one another, and in which
  // order a graph starts two branches is not ours to say (sphere of 8.6e7
  // elements, FP32, ms a step: after 33.1, beside 33.2 or 43.2).  The finest
  // level's bricks are a launch of their own there (and with BF16 storage,
  // whose two-element kernel has no record epilogue).
  ScArgs fin = in;
  int coarse_segs = 0;
  if (in.nseg > 1 && !in.seg[in.nseg - 1].rec_out && (!beside || p.precision == LBM_BF16DEV)) {
    coarse_segs = in.nseg - 1;
    fin.nseg = 1;
    fin.seg[0] = in.seg[in.nseg - 1];
    in.nseg = coarse_segs;
  }
  auto run_outlet = [&](cudaStream_t s) { issued += ops->outlet(Q, out, s); };
  const bool out_branch = out.nlev && !outlet_reads_ghosts;
  if (out_branch) {
    fork(1);
    run_outlet(br.s[1]);
  }
  GffArgs gff = gff_args();
  gff.chain = chain;
  for (int l = l0; l + 1 < n; ++l) {
    const int k = gff.nseg;
    add_gff(gff, l);
    if (gff.nseg > k) launches += 1 + (gff.lev[k].rec_out != nullptr);
  }
  if (gff.nseg) issued += ops->fill_gff(Q, gff, st);
  // Interior bricks beside the GhostFromCoarser fill: queued before it, but
  // after it in FP64, where one-warp blocks of the bricks would fill the slots
  // the fill needs (D2Q9 channel 52 against 40 us)
  const bool early = fin.nseg && beside;
  auto run_early = [&] {
    if (coarse_segs) issued += ops->sc_interior(Q, force, in, br.s[0]);
    timed_launch(timed_level, TK_INTERIOR, [&] { issued += ops->sc_interior(Q, force, fin, br.s[0]); }, br.s[0]);
  };
  const bool fill_first = p.precision == LBM_FP64;
  if (early) {
    fork(0);
    if (!fill_first) run_early();
  }
  GfcArgs gfc = gfc_args();
  gfc.chain = chain;
  if (p.time_mode == LBM_TIME_LINEAR && l0 > 0) {
    if (at_mid_step) at_mid_step(l0 - 1);
    source_moments(l0 - 1, ld[l0 - 1].momA[parity[l0 - 1]], nullptr, SRC_GFF_OUTER);
    add_gfc(gfc, l0, true, false);
  }
  for (int l = l0 + 1; l < n; ++l) add_gfc(gfc, l, false, false);
  launches += gfc.nseg;
  if (gfc.nseg) issued += ops->fill_gfc(Q, gfc, st);
  if (early && fill_first) run_early();
  if (out.nlev && !out_branch) run_outlet(st);
  if (out_branch) join(1);
  timed_launch(timed_level, TK_SC_SPAN, [&] {
    if (fin.nseg && !beside) {
      fork(0);
      if (coarse_segs) issued += ops->sc_interior(Q, force, in, br.s[0]);
      timed_launch(timed_level, TK_INTERIOR, [&] { issued += ops->sc_interior(Q, force, fin, br.s[0]); }, br.s[0]);
    }
    if (rest.nseg) timed_launch(timed_level, TK_BOUNDARY, [&] { issued += ops->sc_rest(Q, force, rest, st); });
    if (rest_fin.nseg) issued += ops->sc_rest(Q, force, rest_fin, st);
    if (fin.nseg) join(0);
  });
  for (int l = l0; l < n; ++l) parity[l] ^= 1;
}

void lbm_ctx::ensure_records() {
  if (recs_valid || dry) return;
  for (int li = 0; li + 1 < nlev; ++li) source_moments(li, ld[li].momA[parity[li]]);
  recs_valid = true;
}

// The recursive step of Sec. 2.2, kernel by kernel on the bound stream (timing
// mode 1, the adjoint's recorded steps, a dry walk of the op sequence).
// Source records (interpolation step 1), two buffers per level: momA[parity]
// holds those of the current state.  The stream-collide writes the records of
// the sources it updates into the other buffer (their state at t + 1), the
// GhostFromFiner fill those of its ghosts at t, and in LINEAR mode the outer
// GhostFromFiner layer, which no stream-collide updates, gets its records at
// t + 1 from its stored state.  The fill at t + 1/2 takes the means of the
// two buffers.
void lbm_ctx::advance(int li) {
  const bool has_finer = li + 1 < nlev;
  const bool linear = p.time_mode == LBM_TIME_LINEAR;
  auto op = [&](int kind, int level) {
    if (hook) hook(kind, level);
    return !dry;
  };
  if (has_finer) {
    if (op(OP_GFF, li)) fill_gff(li);
    // the records of the GhostFromFiner sources: written by the fill
    if (op(OP_MOM_A, li) && ld[li].n_gsrc > 0) ++launches;
    if (op(OP_GFC_A, li + 1)) fill_gfc(li + 1, false, false);
  }
  if (op(OP_SC, li)) stream_collide(li);
  else parity[li] ^= 1;
  if (has_finer) {
    advance(li + 1);
    if (linear) {
      if (op(OP_MOM_B, li)) {
        if (at_mid_step) at_mid_step(li);
        source_moments(li, ld[li].momA[parity[li]], nullptr, SRC_GFF_OUTER);
      }
      if (op(OP_GFC_B, li + 1)) fill_gfc(li + 1, true, false);
    }
    // the remaining substeps (one in acoustic scaling; three with diffusive
    // scaling, whose four ghost layers filled at t last all four)
    for (int k = 1; k < time_ratio(p.time_mode); ++k) advance(li + 1);
  }
}

void lbm_ctx::set_priority() {
  int bound = 0, least = 0, greatest = 0;
  if (cudaStreamGetPriority(st, &bound) != cudaSuccess || cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) {
    cudaGetLastError();
    bound = greatest = 0;
  }
  const StepPriority p = step_priority(bound, greatest);
  if (p.bricks != prio.bricks || p.chain != prio.chain) drop_streams();
  prio = p;
}

bool lbm_ctx::make_branches() {
  if (br.s[0]) return br.ok;
  br.ok = true;
  for (int b = 0; b < 2; ++b) {
    br.ok = br.ok && cudaStreamCreateWithPriority(&br.s[b], cudaStreamNonBlocking,
                                                  b == 0 ? prio.bricks : prio.chain) == cudaSuccess;
    for (cudaEvent_t* e : {&br.fork[b], &br.join[b]})
      br.ok = br.ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
  }
  if (!br.ok) cudaGetLastError();
  return br.ok;
}

const lbm_ctx::StepGraph* lbm_ctx::step_graph(int nsteps) {
  for (const StepGraph& g : graphs)
    if (g.parity == parity && g.steps == nsteps) return &g;
  if (!cap_stream && cudaStreamCreateWithPriority(&cap_stream, cudaStreamNonBlocking, prio.chain) != cudaSuccess) {
    cudaGetLastError();
    graphs_on = false;
    return nullptr;
  }
  // levels batched by instant (up to kMaxBatch of them); without branch
  // streams, or with more levels, the captured steps are the recursion's
  const bool batched = can_batch();
  // capture on a private stream (the bound stream may be the legacy default
  // stream, which cannot be captured); host bookkeeping is restored afterwards
  const std::vector<int> p0 = parity;
  const int64_t l0 = launches, i0 = issued;
  if (timing == 2) {
    // events for the finest level's stream-collide launches and their span
    // (up to four pairs per substep, m^(nlev-1) substeps per coarse step, m
    // the time-step ratio), made before the capture begins (at most 2^16;
    // further ones are made as they are needed)
    int64_t nev = (int64_t)nsteps * 4 * 2;
    for (int li = 1; li < nlev && nev < (1 << 16); ++li) nev *= time_ratio(p.time_mode);
    for (int64_t k = 0; k < std::min<int64_t>(nev, 1 << 16); ++k) event_pool.push_back(get_event());
  }
  const size_t t0 = timed.size();
  cudaStream_t user = st;
  st = cap_stream;
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamBeginCapture(cap_stream, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    capturing = true;
    for (int k = 0; k < nsteps; ++k) {
      if (batched) step_batched();
      else advance(0);
    }
    capturing = false;
    e = cudaStreamEndCapture(cap_stream, &graph);
  }
  st = user;
  std::vector<Timed> gt(timed.begin() + t0, timed.end());
  timed.resize(t0);
  const int64_t nl = launches - l0, ni = issued - i0;
  launches = l0;
  issued = i0;
  // two steps bring every level back to its buffer; one step flips the
  // coarsest level's (the finer levels take an even number of substeps)
  std::vector<int> expect = p0;
  if (nsteps == 1) expect[0] ^= 1;
  const std::vector<int> p1 = parity;
  const bool same = p1 == expect;
  parity = p0;
  cudaGraphExec_t exec = nullptr;
  if (e == cudaSuccess && graph && same)
    e = cudaGraphInstantiate(&exec, graph, batched && prioritised() ? cudaGraphInstantiateFlagUseNodePriority : 0);
  if (graph) cudaGraphDestroy(graph);
  if (e != cudaSuccess || !exec || !same) {
    cudaGetLastError();
    for (auto& t : gt) {
      event_pool.push_back(t.a);
      event_pool.push_back(t.b);
    }
    (nsteps > 2 ? long_graphs_on : graphs_on) = false;
    return nullptr;
  }
  graphs.push_back({p0, p1, nsteps, exec, nl, ni, std::move(gt)});
  return &graphs.back();
}

// ---------------------------------------------------------------- internal accessors
namespace lbm {

lbm_status reduce_plan(lbm_ctx* c, ReducePlan* plan) {
  if (!c || !plan) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "reduction before lbm_bind");
  plan->ops = c->ops;
  plan->Q = c->Q;
  plan->stream = c->st;
  plan->workspace = c->ws;
  ReduceArgs& a = plan->args;
  a = ReduceArgs{};
  a.force = c->force_ptr();
  a.Ntot = c->M.Ntot;
  a.rho_off = c->rho_off;
  a.rho0 = c->p.rho0;
  a.nseg = c->nlev;
  const int d = c->d;
  for (int li = 0; li < c->nlev; ++li) {
    const HostLevel& H = c->M.lv[li];
    ReduceLevel& l = a.lev[li];
    l.pdf = c->cur(li);
    l.begin = H.base + H.oF;
    l.end = H.base + H.oF + H.nF;
    l.vol = std::ldexp(1.0, -d * li);
    // diffusive scaling: mass, momentum and kinetic energy in the coarsest
    // level's units (a lattice velocity of level li is 2^li of the
    // coarsest's), forces in the finest level's (a force unit goes with
    // dx^(d+1) / dt^2)
    const double us = 1.0 / level_velocity_ratio(li, c->p.time_mode);
    l.vol_m = l.vol * us;
    l.vol_k = l.vol * us * us;
    l.r_scale = us * us;
    l.obs_elem = c->at<int32_t>(c->oObsElem) + H.obs_begin;
    l.obs_dir = c->at<int8_t>(c->oObsDir) + H.obs_begin;
    l.obs_a = c->at<int32_t>(c->oObsA) + H.obs_begin;
    l.obs_q = c->at<double>(c->oObsQ) + H.obs_begin;
    l.obs_n = H.obs_end - H.obs_begin;
    l.fscale = std::ldexp(1.0, (c->p.time_mode == LBM_TIME_DIFFUSIVE ? d - 3 : d - 1) * (c->nlev - 1 - li));
  }
  return LBM_OK;
}

lbm_status set_error(lbm_ctx* c, lbm_status s, const std::string& msg) { return c->fail(s, msg); }

void count_launches(lbm_ctx* c, int64_t level_kernels, int64_t issued) {
  c->launches += level_kernels;
  c->issued += issued;
}

}  // namespace lbm

// ---------------------------------------------------------------- C ABI
extern "C" {

lbm_status lbm_build_mesh(const int64_t* tree_ids, const int8_t* levels, int64_t n, const lbm_params* params,
                          lbm_ctx** out) {
  if (!out || !params) return LBM_ERR_ARG;
  *out = nullptr;
  lbm_ctx* c = new (std::nothrow) lbm_ctx();
  if (!c) return LBM_ERR_OOM;
  c->p = *params;
  if (params->precision == LBM_FP64) c->ops = ops_fp64();
  else if (params->precision == LBM_FP32DEV) c->ops = ops_fp32dev();
  else if (params->precision == LBM_BF16DEV) c->ops = ops_bf16dev();
  else {
    c->err = "bad precision";
    *out = c;
    return LBM_ERR_ARG;
  }
  if (params->outlet != LBM_OUTLET_LINEAR && params->outlet != LBM_OUTLET_ZERO_GRADIENT) {
    c->err = "bad outlet extrapolation";
    *out = c;
    return LBM_ERR_ARG;
  }
  if (params->check_every < 0 || !(params->mass_band >= 0.0) || !std::isfinite(params->mass_band)) {
    c->err = "check_every must be >= 0 and mass_band finite and >= 0";
    *out = c;
    return LBM_ERR_ARG;
  }
  if (params->adjoint_tape < 0 || params->adjoint_tape > 2) {
    c->err = "adjoint_tape must be 0, 1 or 2";
    *out = c;
    return LBM_ERR_ARG;
  }
  lbm_status s;
  try {
    s = build_host_mesh(tree_ids, levels, n, c->p, &c->M, &c->err);
  } catch (const std::bad_alloc&) {
    c->err = "host allocation failed";
    s = LBM_ERR_OOM;
  }
  *out = c;
  if (s != LBM_OK) return s;
  c->Q = c->M.Q;
  c->d = c->M.d;
  c->nS = c->M.nS;
  c->nlev = (int)c->M.lv.size();
  c->rho_off = params->precision == LBM_FP64 ? 0.0 : params->rho0;
  int cc[kQmax][3];
  double w[kQmax];
  host_lattice(c->Q, cc, w);
  for (int i = 0; i < c->Q; ++i) {
    double cu = 0;
    for (int a = 0; a < c->d; ++a) cu += cc[i][a] * params->u_in[a];
    c->inlet[i] = 6.0 * w[i] * params->rho0 * cu;
  }
  c->layout();
  c->parity.assign(c->nlev, 0);
  return LBM_OK;
}

lbm_status lbm_mesh_info(const lbm_ctx* c, int64_t* info, int32_t cap, int32_t* nlevels) {
  if (!c || !info) return LBM_ERR_ARG;
  int n = 0;
  for (const HostLevel& H : c->M.lv) {
    if (n >= cap) break;
    int64_t r[10] = {H.L, H.nF, H.nC, H.nG1, H.nG2, H.N, H.out_end - H.out_begin, H.obs_end - H.obs_begin,
                     H.nB, H.nBb};
    std::memcpy(info + 10 * n, r, sizeof(r));
    ++n;
  }
  if (nlevels) *nlevels = (int32_t)c->M.lv.size();
  return LBM_OK;
}

lbm_status lbm_obstacle_links(const lbm_ctx* c, int64_t* elem, int8_t* dir, int64_t cap, int64_t* n) {
  if (!c || !n || cap < 0 || (cap > 0 && (!elem || !dir))) return LBM_ERR_ARG;
  const HostMesh& m = c->M;
  const int64_t cnt = (int64_t)m.obs_elem.size();
  *n = cnt;
  if (cap == 0 || cnt == 0) return LBM_OK;
  // global element slot -> caller index
  std::vector<int64_t> user_of(m.Ntot, -1);
  for (int64_t k = 0; k < m.n_user; ++k) user_of[m.uslot[k]] = k;
  for (int64_t l = 0; l < std::min(cap, cnt); ++l) {
    elem[l] = user_of[m.obs_elem[l]];
    dir[l] = m.obs_dir[l];
  }
  return LBM_OK;
}

lbm_status lbm_set_link_q(lbm_ctx* c, const double* q, int64_t n) {
  if (!c || (n > 0 && !q)) return LBM_ERR_ARG;
  if (!c->p.bouzidi) return c->fail(LBM_ERR_STATE, "params.bouzidi is 0");
  HostMesh& m = c->M;
  if (n != (int64_t)m.obs_elem.size()) return c->fail(LBM_ERR_ARG, "n differs from the obstacle link count");
  for (int64_t l = 0; l < n; ++l)
    if (!(q[l] > 0.0 && q[l] <= 1.0)) return c->fail(LBM_ERR_ARG, "wall distance outside (0, 1]");
  for (int64_t l = 0; l < n; ++l) {
    m.obs_q[l] = q[l];
    if (m.obs_side[l] >= 0) m.out_q[m.obs_side[l]] = q[l];
  }
  if (!c->bound) return LBM_OK;  // uploaded by lbm_bind
  lbm_status s = c->cuda_check(
      cudaMemcpyAsync(c->ws + c->oObsQ, m.obs_q.data(), m.obs_q.size() * 8, cudaMemcpyHostToDevice, c->st), "link q");
  if (s == LBM_OK)
    s = c->cuda_check(
        cudaMemcpyAsync(c->ws + c->oOutQ, m.out_q.data(), m.out_q.size() * 8, cudaMemcpyHostToDevice, c->st), "link q");
  if (s == LBM_OK) s = c->cuda_check(cudaStreamSynchronize(c->st), "link q");
  return s;
}

lbm_status lbm_device_bytes(const lbm_ctx* c, uint64_t* bytes) {
  if (!c || !bytes || !c->ops || c->M.lv.empty()) return LBM_ERR_ARG;
  *bytes = c->bytes;
  return LBM_OK;
}

lbm_status lbm_bind(lbm_ctx* c, void* ws, uint64_t bytes, void* stream) {
  if (!c || !ws) return LBM_ERR_ARG;
  if (c->M.lv.empty()) return c->fail(LBM_ERR_STATE, "no mesh");
  if (bytes < c->bytes) return c->fail(LBM_ERR_ARG, "device workspace too small");
  if (reinterpret_cast<uintptr_t>(ws) % kAlign) return c->fail(LBM_ERR_ARG, "device workspace not 256-byte aligned");
  c->drop_graphs();  // captured steps point into the previous workspace
  c->ws = static_cast<char*>(ws);
  c->st = static_cast<cudaStream_t>(stream);
  c->set_priority();
  c->reset_state_buffers();
  c->pinned_result();
  const HostMesh& m = c->M;
  auto up = [&](size_t off, const void* src, size_t b) -> lbm_status {
    if (b == 0) return LBM_OK;
    return c->cuda_check(cudaMemcpyAsync(c->ws + off, src, b, cudaMemcpyHostToDevice, c->st), "upload");
  };
  lbm_status s = up(c->oNbr, m.nbr.data(), m.nbr.size() * 4);
  if (s == LBM_OK) s = up(c->oBrickNb, m.brick_nb.data(), m.brick_nb.size() * 4);
  if (s == LBM_OK) s = up(c->oBrickTab, m.brick_tab.data(), m.brick_tab.size() * 2);
  if (s == LBM_OK) s = up(c->oInletS, m.inlet_s.data(), m.inlet_s.size() * 8);
  if (s == LBM_OK) s = up(c->oOutQ, m.out_q.data(), m.out_q.size() * 8);
  if (s == LBM_OK) s = up(c->oObsA, m.obs_a.data(), m.obs_a.size() * 4);
  if (s == LBM_OK) s = up(c->oObsQ, m.obs_q.data(), m.obs_q.size() * 8);
  for (int li = 0; li < c->nlev && s == LBM_OK; ++li) {
    const HostLevel& H = m.lv[li];
    s = up(c->ld[li].gff_child0, H.gff_child0.data(), H.gff_child0.size() * 4);
    if (s == LBM_OK) s = up(c->ld[li].gfc_src, H.gfc_src.data(), H.gfc_src.size() * 4);
    if (s == LBM_OK) s = up(c->ld[li].gfc_oct, H.gfc_oct.data(), H.gfc_oct.size());
    if (s == LBM_OK) s = up(c->ld[li].src_elem, H.src_elem.data(), H.src_elem.size() * 4);
    if (s == LBM_OK) s = up(c->ld[li].gsrc_elem, H.gsrc_elem.data(), H.gsrc_elem.size() * 4);
    if (s == LBM_OK) s = up(c->ld[li].gsrc_rec, H.gsrc_rec.data(), H.gsrc_rec.size() * 4);
  }
  if (s == LBM_OK) s = up(c->oSrcMask, m.src_mask.data(), m.src_mask.size() * 4);
  if (s == LBM_OK) s = up(c->oSrcFirst, m.src_first.data(), m.src_first.size() * 4);
  if (s == LBM_OK) s = up(c->oOutElem, m.out_elem.data(), m.out_elem.size() * 4);
  if (s == LBM_OK) s = up(c->oOutA, m.out_a.data(), m.out_a.size() * 4);
  if (s == LBM_OK) s = up(c->oOutB, m.out_b.data(), m.out_b.size() * 4);
  if (s == LBM_OK) s = up(c->oOutDir, m.out_dir.data(), m.out_dir.size());
  if (s == LBM_OK) s = up(c->oOutKind, m.out_kind.data(), m.out_kind.size());
  if (s == LBM_OK) s = up(c->oObsElem, m.obs_elem.data(), m.obs_elem.size() * 4);
  if (s == LBM_OK) s = up(c->oObsDir, m.obs_dir.data(), m.obs_dir.size());
  if (s == LBM_OK) s = up(c->oUslot, m.uslot.data(), m.uslot.size() * 4);
  if (s == LBM_OK) s = up(c->oUlev, m.ulev.data(), m.ulev.size());
  if (s == LBM_OK) s = up(c->oSlotUser, m.slot_user.data(), m.slot_user.size() * 4);
  if (s != LBM_OK) return s;
  if (c->p.use_force) {
    s = c->cuda_check(cudaMemsetAsync(c->ws + c->oF, 0, (size_t)c->d * m.Ntot * c->ops->compute_bytes, c->st),
                      "force clear");
    if (s != LBM_OK) return s;
  }
  for (size_t off : {c->oA, c->oB}) {
    FillArgs f{c->ws + off, m.Ntot, c->p.rho0, c->rho_off};
    c->ops->fill_rest(c->Q, f, c->st);
    count_launches(c, 1, 1);
  }
  s = c->launched("bind");
  if (s == LBM_OK) s = c->cuda_check(cudaStreamSynchronize(c->st), "bind sync");
  if (s != LBM_OK) return s;
  std::fill(c->parity.begin(), c->parity.end(), 0);
  c->reset_check();
  c->bound = true;
  return LBM_OK;
}

lbm_status lbm_init(lbm_ctx* c, const double* rho, const double* u, const double* S, const double* df) {
  if (!c || !rho || !u) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_init before lbm_bind");
  const int64_t n = c->M.n_user;
  const int d = c->d, nS = c->nS, Q = c->Q;
  // Every level starts in A.  The chunks are computed in caller order into B
  // (coalesced writes, B holds nothing that survives an init), then placed
  // into the element slots of A in slot order, and B is reset to rest.
  // The staging area is used as two halves: the host copies of one half-chunk
  // (on the context's copy stream) overlap the init kernel of the other.
  std::fill(c->parity.begin(), c->parity.end(), 0);
  c->reset_check();
  const bool two = c->copy_stream_ready();
  const int64_t CH = two ? (c->chunk + 1) / 2 : c->chunk;
  const int64_t per = 1 + d + nS + Q;  // staged doubles per element
  cudaStream_t cs = two ? c->copy_st : c->st;
  if (two) {
    // the staging area may still be read by earlier work on the bound stream
    cudaEventRecord(c->copy_ev[2], c->st);
    cudaStreamWaitEvent(cs, c->copy_ev[2], 0);
  }
  int64_t i = 0;
  for (int64_t first = 0; first < n; first += CH, ++i) {
    const int64_t cnt = std::min(CH, n - first);
    const int half = two ? (int)(i & 1) : 0;
    double* sr = c->at<double>(c->oStage) + (size_t)half * CH * per;
    double* su = sr + CH;
    double* sS = su + CH * d;
    double* sdf = sS + CH * nS;
    // this half's previous init kernel has read it
    if (two && i >= 2) cudaStreamWaitEvent(cs, c->copy_ev[half], 0);
    lbm_status s = c->cuda_check(cudaMemcpyAsync(sr, rho + first, cnt * 8, cudaMemcpyHostToDevice, cs), "init copy");
    if (s == LBM_OK)
      s = c->cuda_check(cudaMemcpyAsync(su, u + first * d, cnt * d * 8, cudaMemcpyHostToDevice, cs), "init copy");
    if (s == LBM_OK && S)
      s = c->cuda_check(cudaMemcpyAsync(sS, S + first * nS, cnt * nS * 8, cudaMemcpyHostToDevice, cs), "init copy");
    if (s == LBM_OK && df)
      s = c->cuda_check(cudaMemcpyAsync(sdf, df + first * Q, cnt * Q * 8, cudaMemcpyHostToDevice, cs), "init copy");
    if (s != LBM_OK) return s;
    if (two) {
      cudaEventRecord(c->copy_ev[3], cs);
      cudaStreamWaitEvent(c->st, c->copy_ev[3], 0);
    }
    InitArgs a{};
    a.temp = c->at(c->oB);
    a.ulev = c->at<uint8_t>(c->oUlev);
    a.rho = sr;
    a.u = su;
    a.S = S ? sS : nullptr;
    a.df = df ? sdf : nullptr;
    a.first = first;
    a.cnt = cnt;
    a.n_user = n;
    for (int li = 0; li < c->nlev; ++li) a.omega[li] = c->M.lv[li].omega;
    a.rho_off = c->rho_off;
    c->ops->init(Q, a, c->st);
    count_launches(c, 1, 1);
    if (two) cudaEventRecord(c->copy_ev[half], c->st);
  }
  PlaceArgs pl{c->at(c->oB), c->at(c->oA), c->at<int32_t>(c->oSlotUser), n, c->M.Ntot};
  c->ops->init_place(Q, pl, c->st);
  count_launches(c, 1, 1);
  FillArgs f{c->at(c->oB), c->M.Ntot, c->p.rho0, c->rho_off};
  c->ops->fill_rest(Q, f, c->st);
  count_launches(c, 1, 1);
  lbm_status s = c->launched("init");
  if (s == LBM_OK) s = c->cuda_check(cudaStreamSynchronize(c->st), "init sync");
  return s;
}

lbm_status lbm_set_force(lbm_ctx* c, const double* F) {
  if (!c || !F) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_set_force before lbm_bind");
  if (!c->p.use_force) return c->fail(LBM_ERR_STATE, "params.use_force is 0");
  const int64_t n = c->M.n_user, CH = c->chunk;
  double* sf = c->at<double>(c->oStage);
  for (int64_t first = 0; first < n; first += CH) {
    const int64_t cnt = std::min(CH, n - first);
    lbm_status s = c->cuda_check(
        cudaMemcpyAsync(sf, F + first * c->d, cnt * c->d * 8, cudaMemcpyHostToDevice, c->st), "force copy");
    if (s != LBM_OK) return s;
    ForceArgs a{c->at(c->oF), c->at<int32_t>(c->oUslot), sf, first, cnt, c->M.Ntot, c->d};
    launch_scatter_force(c->p.precision == LBM_FP64, a, c->st);
    count_launches(c, 1, 1);
  }
  c->recs_valid = false;
  lbm_status s = c->launched("set_force");
  if (s == LBM_OK) s = c->cuda_check(cudaStreamSynchronize(c->st), "force sync");
  return s;
}

static lbm_status step_run(lbm_ctx* c, int64_t n_coarse);

// the FP64 reductions of the current state into out[8] (host), synchronising
static lbm_status reduce_to_host(lbm_ctx* c, double out[8]) {
  // the per-level arguments come from the one plan builder (also used by
  // lbm_reduce_noalloc); only the partial rows differ
  ReducePlan plan;
  lbm_status ps = reduce_plan(c, &plan);
  if (ps != LBM_OK) return ps;
  plan.args.partial = c->at<double>(c->oPartial);
  const unsigned rows = c->ops->reduce(c->Q, plan.args, c->st);
  // the result goes straight to pinned host memory (a copy of 64 bytes costs
  // about 8 us more), or through the workspace where there is none
  double* pinned = c->result_host;
  FinalArgs fa{c->at<double>(c->oPartial), (int64_t)rows, pinned ? pinned : c->at<double>(c->oRed)};
  launch_final_reduce(fa, c->st);
  count_launches(c, c->nlev + 1, 2);  // a level's reduction counts as a level kernel
  lbm_status s = c->launched("reduce");
  if (s == LBM_OK && !pinned)
    s = c->cuda_check(cudaMemcpyAsync(out, c->at(c->oRed), 64, cudaMemcpyDeviceToHost, c->st), "reduce copy");
  if (s == LBM_OK) s = c->cuda_check(cudaStreamSynchronize(c->st), "reduce sync");
  if (s == LBM_OK && pinned) std::memcpy(out, pinned, 64);
  return s;
}

// the mass check of params.check_every: finite, and within mass_band of the
// reference mass when a band is set
static lbm_status check_mass(lbm_ctx* c, bool reference) {
  double r[8];
  lbm_status s = reduce_to_host(c, r);
  if (s != LBM_OK) return s;
  const double m = r[0];
  char buf[160];
  if (!std::isfinite(m)) {
    std::snprintf(buf, sizeof buf, "mass check after %lld coarse steps: mass is not finite (%g)",
                  (long long)c->steps_done, m);
    return c->fail(LBM_ERR_NUMERIC, buf);
  }
  if (reference) {
    c->mass_ref = m;
    c->mass_ref_valid = true;
    return LBM_OK;
  }
  if (c->p.mass_band > 0.0 && std::fabs(m / c->mass_ref - 1.0) > c->p.mass_band) {
    std::snprintf(buf, sizeof buf, "mass check after %lld coarse steps: mass %.17g outside %g of %.17g",
                  (long long)c->steps_done, m, c->p.mass_band, c->mass_ref);
    return c->fail(LBM_ERR_NUMERIC, buf);
  }
  return LBM_OK;
}

// n_coarse coarse steps with no check in between
lbm_status lbm_ctx::run_steps(int64_t n_coarse) { return step_run(this, n_coarse); }

static lbm_status step_run(lbm_ctx* c, int64_t n_coarse) {
  int64_t k = 0;
  if (n_coarse > 0) c->ensure_records();  // outside any capture
  // pairs of coarse steps replay a captured two-step graph and a remaining
  // single step a one-step graph (small meshes, later, longer ones); timed
  // steps (mode 1) are issued one kernel at a time
  if (c->graphs_on && c->timing != 1 && !c->hook && !c->dry) {
    while (k < n_coarse) {
      const int64_t left = n_coarse - k;
      const bool longer = left >= kLongGraphSteps && c->long_graphs();
      const lbm_ctx::StepGraph* g = longer ? c->step_graph(kLongGraphSteps) : nullptr;
      if (!g) g = c->step_graph(left >= 2 ? 2 : 1);
      if (!g) break;
      lbm_status s = c->cuda_check(cudaGraphLaunch(g->exec, c->st), "graph launch");
      if (s != LBM_OK) return s;
      count_launches(c, g->launches, g->issued);
      c->parity = g->end;
      c->last_graph = (int)(g - c->graphs.data());
      c->graph_unread = true;
      c->graph_steps += g->steps;
      k += g->steps;
    }
  }
  for (; k < n_coarse; ++k) c->coarse_step();
  return c->launched("step");
}

lbm_status lbm_step(lbm_ctx* c, int64_t n_coarse) {
  if (!c || n_coarse < 0) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_step before lbm_bind");
  const int64_t M = c->p.check_every;
  if (M <= 0) {
    c->steps_done += n_coarse;
    return step_run(c, n_coarse);
  }
  // the optional mass check: after every M-th coarse step, counted across calls
  if (!c->mass_ref_valid && n_coarse > 0) {
    lbm_status s = check_mass(c, true);
    if (s != LBM_OK) return s;
  }
  int64_t done = 0;
  while (done < n_coarse) {
    const int64_t chunk = std::min(n_coarse - done, M - c->steps_since_check);
    lbm_status s = step_run(c, chunk);
    if (s != LBM_OK) return s;
    done += chunk;
    c->steps_done += chunk;
    c->steps_since_check += chunk;
    if (c->steps_since_check == M) {
      c->steps_since_check = 0;
      s = check_mass(c, false);
      if (s != LBM_OK) return s;
    }
  }
  return LBM_OK;
}

lbm_status lbm_fill_ghosts(lbm_ctx* c) {
  if (!c) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_fill_ghosts before lbm_bind");
  for (int li = 0; li + 1 < c->nlev; ++li) {
    c->fill_gff(li);
    c->source_moments(li, c->ld[li].momA[c->parity[li]]);
    c->fill_gfc(li + 1, false, true);
  }
  c->recs_valid = true;  // every record now holds the current state's moments
  return c->launched("fill_ghosts");
}

// Makes the pages of a large host output present, on all cores, while the GPU
// works on the first chunk: a device-to-host copy into memory that was never
// written stops at every page (64 KiB here) for the system to clear it, which
// took 75 MB from 0.4 to 3.2 ms.  One byte of each page is written; the call
// overwrites the whole array.
static void touch_pages(void* p, size_t bytes) {
  if (!p || bytes < ((size_t)4 << 20)) return;
  // pinned memory has its pages; device memory, or memory that the runtime
  // cannot tell (the context is lost), is for the copy to refuse
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess || at.type != cudaMemoryTypeUnregistered) {
    cudaGetLastError();
    return;
  }
  const size_t page = (size_t)std::max(4096l, sysconf(_SC_PAGESIZE));
  volatile char* b = static_cast<volatile char*>(p);
  const int64_t n = (int64_t)((bytes + page - 1) / page);
#pragma omp parallel for schedule(static)
  for (int64_t k = 0; k < n; ++k) b[(size_t)k * page] = 0;
}

static lbm_status out_chunks(lbm_ctx* c, double* rho, double* u, double* S, double* f) {
  const int64_t n = c->M.n_user;
  const int d = c->d, nS = c->nS, Q = c->Q;
  // Two halves of the staging area: the copy of one chunk to the host (on the
  // copy stream) beside the kernel of the next, where the chunks' copies are
  // long against the 10 us that each costs (moments of 1.5e5 D3Q19 elements in
  // four chunks 268 us, in one 219; of 4.9e5 elements 424 and 609 us, of
  // 1.08e7 5.4 ms in halves of the staging area and 12.5 in whole chunks, most
  // of both from the kernel's fewer FP64 instructions).
  const bool two = n >= (1 << 18) && c->copy_stream_ready();
  const int64_t CH = two ? std::min((c->chunk + 1) / 2, std::max<int64_t>((n + 3) / 4, 1 << 17)) : c->chunk;
  const int64_t per = 1 + d + nS + Q;  // staged doubles per element
  cudaStream_t cs = two ? c->copy_st : c->st;
  if (two) {
    // the staging area may still be read by earlier work on the bound stream
    cudaEventRecord(c->copy_ev[2], c->st);
    cudaStreamWaitEvent(cs, c->copy_ev[2], 0);
  }
  OutArgs a{};
  a.A = c->at(c->oA);
  a.B = c->at(c->oB);
  a.force = c->force_ptr();
  a.uslot = c->at<int32_t>(c->oUslot);
  a.ulev = c->at<uint8_t>(c->oUlev);
  a.parity = c->parity_mask();
  a.Ntot = c->M.Ntot;
  for (int li = 0; li < c->nlev; ++li) a.rx[li] = make_relax(Q, c->M.lv[li].omega);
  a.rho_off = c->rho_off;
  lbm_status s = LBM_OK;
  const int64_t chunks = (n + CH - 1) / CH;
  auto stage = [&](int64_t i) { return c->at<double>(c->oStage) + (size_t)(two ? i & 1 : 0) * CH * per; };
  auto compute = [&](int64_t i) {
    // the half's previous copies are done
    if (two && i >= 2) cudaStreamWaitEvent(c->st, c->copy_ev[i & 1], 0);
    double* sr = stage(i);
    a.rho = rho ? sr : nullptr;
    a.u = u ? sr + CH : nullptr;
    a.S = S ? sr + CH * (1 + d) : nullptr;
    a.f = f ? sr + CH * (1 + d + nS) : nullptr;
    a.first = i * CH;
    a.cnt = std::min(CH, n - a.first);
    c->ops->out(Q, a, c->st);
    count_launches(c, 1, 1);
    if (two) cudaEventRecord(c->copy_ev[2 + (i & 1)], c->st);
  };
  compute(0);
  touch_pages(rho, (size_t)n * 8);
  touch_pages(u, (size_t)n * d * 8);
  touch_pages(S, (size_t)n * nS * 8);
  touch_pages(f, (size_t)n * Q * 8);
  for (int64_t i = 0; i < chunks && s == LBM_OK; ++i) {
    // a copy to pageable memory may hold this thread, so the next chunk's
    // kernel is launched before it
    if (two && i + 1 < chunks) compute(i + 1);
    if (two) cudaStreamWaitEvent(cs, c->copy_ev[2 + (i & 1)], 0);
    const int64_t first = i * CH, cnt = std::min(CH, n - first);
    const double* sr = stage(i);
    auto down = [&](double* dst, const double* src, size_t b) {
      if (s == LBM_OK) s = c->cuda_check(cudaMemcpyAsync(dst, src, b, cudaMemcpyDeviceToHost, cs), "output copy");
    };
    if (rho) down(rho + first, sr, cnt * 8);
    if (u) down(u + first * d, sr + CH, cnt * d * 8);
    if (S) down(S + first * nS, sr + CH * (1 + d), cnt * nS * 8);
    if (f) down(f + first * Q, sr + CH * (1 + d + nS), cnt * Q * 8);
    if (two) cudaEventRecord(c->copy_ev[i & 1], cs);
    else if (i + 1 < chunks) compute(i + 1);
  }
  if (s == LBM_OK) s = c->launched("output");
  // both streams idle: the staging area and the host arrays are free
  const lbm_status e = c->cuda_check(cudaStreamSynchronize(c->st), "output sync");
  const lbm_status e2 = c->cuda_check(cudaStreamSynchronize(cs), "output sync");
  return s != LBM_OK ? s : e != LBM_OK ? e : e2;
}

lbm_status lbm_moments(lbm_ctx* c, double* rho, double* u, double* S) {
  if (!c) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_moments before lbm_bind");
  return out_chunks(c, rho, u, S, nullptr);
}

lbm_status lbm_get_state(lbm_ctx* c, double* f) {
  if (!c || !f) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_get_state before lbm_bind");
  return out_chunks(c, nullptr, nullptr, nullptr, f);
}

lbm_status lbm_set_state(lbm_ctx* c, const double* f) {
  if (!c || !f) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_set_state before lbm_bind");
  const int64_t n = c->M.n_user, CH = c->chunk;
  double* sf = c->at<double>(c->oStage);
  c->reset_check();
  for (int64_t first = 0; first < n; first += CH) {
    const int64_t cnt = std::min(CH, n - first);
    lbm_status s = c->cuda_check(
        cudaMemcpyAsync(sf, f + first * c->Q, cnt * c->Q * 8, cudaMemcpyHostToDevice, c->st), "state copy");
    if (s != LBM_OK) return s;
    SetStateArgs a{c->at(c->oA), c->at(c->oB), c->at<int32_t>(c->oUslot), c->at<uint8_t>(c->oUlev),
                   c->parity_mask(), sf, first, cnt, c->M.Ntot, c->rho_off};
    c->ops->set_state(c->Q, a, c->st);
    count_launches(c, 1, 1);
  }
  lbm_status s = c->launched("set_state");
  if (s == LBM_OK) s = c->cuda_check(cudaStreamSynchronize(c->st), "state sync");
  return s;
}

lbm_status lbm_reduce(lbm_ctx* c, double out[8]) {
  if (!c || !out) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_reduce before lbm_bind");
  return reduce_to_host(c, out);
}

lbm_status lbm_ghost_count(const lbm_ctx* c, int64_t* n) {
  if (!c || !n) return LBM_ERR_ARG;
  int64_t t = 0;
  for (const HostLevel& H : c->M.lv) t += H.nC + H.nG1 + H.nG2;
  *n = t;
  return LBM_OK;
}

lbm_status lbm_get_ghosts(lbm_ctx* c, int64_t* info, double* f) {
  if (!c || !info || !f) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_get_ghosts before lbm_bind");
  const int Q = c->Q;
  int64_t row = 0;
  double* stage = c->at<double>(c->oStage);
  for (int li = 0; li < c->nlev; ++li) {
    const HostLevel& H = c->M.lv[li];
    const int64_t ng = H.nC + H.nG1 + H.nG2;
    for (int64_t k = 0; k < ng; ++k) {
      int64_t* r = info + 6 * (row + k);
      r[0] = H.L;
      r[1] = k < H.nC ? 1 : 2;
      r[2] = H.ghost_layer[k];
      for (int a = 0; a < 3; ++a) r[3 + a] = H.ghost_xyz[3 * k + a];
    }
    const int64_t seg_first[3] = {H.base + H.oC, H.base + H.oG1, H.base + H.oG2};
    const int64_t seg_cnt[3] = {H.nC, H.nG1, H.nG2};
    for (int sgi = 0; sgi < 3; ++sgi) {
      for (int64_t done = 0; done < seg_cnt[sgi]; done += c->chunk) {
        const int64_t cnt = std::min<int64_t>(c->chunk, seg_cnt[sgi] - done);
        GatherGhostArgs a{c->cur(li), seg_first[sgi] + done, cnt, c->M.Ntot, stage, c->rho_off};
        c->ops->gather_ghosts(Q, a, c->st);
        count_launches(c, 1, 1);
        lbm_status s = c->launched("ghosts");
        if (s == LBM_OK)
          s = c->cuda_check(cudaMemcpyAsync(f + (row + done) * Q, stage, cnt * Q * 8, cudaMemcpyDeviceToHost, c->st),
                            "ghost copy");
        if (s == LBM_OK) s = c->cuda_check(cudaStreamSynchronize(c->st), "ghost sync");
        if (s != LBM_OK) return s;
      }
      row += seg_cnt[sgi];
    }
  }
  return LBM_OK;
}

lbm_status lbm_sfc_partition(const int64_t* tree_ids, int64_t n, int32_t d, int32_t nparts, int64_t* order,
                             int64_t* weights, int64_t* cumulative, int32_t* part) {
  std::string msg;
  return sfc_partition(tree_ids, n, d, nparts, order, weights, cumulative, part, &msg);
}

lbm_status lbm_kernel_launches(const lbm_ctx* c, int64_t* count) {
  if (!c || !count) return LBM_ERR_ARG;
  *count = c->launches;
  return LBM_OK;
}

lbm_status lbm_launches(const lbm_ctx* c, int64_t* count) {
  if (!c || !count) return LBM_ERR_ARG;
  *count = c->issued;
  return LBM_OK;
}

lbm_status lbm_timing_enable(lbm_ctx* c, int32_t mode) {
  if (!c) return LBM_ERR_ARG;
  if (mode < 0 || mode > 2) return c->fail(LBM_ERR_ARG, "timing mode must be 0, 1 or 2");
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_timing_enable before lbm_bind");
  lbm_status s = c->cuda_check(cudaStreamSynchronize(c->st), "timing sync");
  c->recycle_timed();
  // graphs captured with events (mode 2) and without them are not interchangeable
  if ((mode == 2) != (c->timing == 2)) c->drop_graphs();
  c->graph_unread = false;
  c->timing = mode;
  return s;
}

lbm_status lbm_timing_read(lbm_ctx* c, int64_t* launches, double* ms, int32_t cap) {
  if (!c || !launches || !ms) return LBM_ERR_ARG;
  if (!c->bound) return c->fail(LBM_ERR_STATE, "lbm_timing_read before lbm_bind");
  lbm_status s = c->cuda_check(cudaStreamSynchronize(c->st), "timing sync");
  if (s != LBM_OK) return s;
  for (int k = 0; k < cap; ++k) {
    launches[k] = 0;
    ms[k] = 0.0;
  }
  auto add = [&](const lbm_ctx::Timed& t) {
    float e = 0.f;
    if (s == LBM_OK) s = c->cuda_check(cudaEventElapsedTime(&e, t.a, t.b), "timing read");
    const int row = kTimedKinds * t.li + t.kernel;
    if (s == LBM_OK && row < cap) {
      launches[row] += 1;
      ms[row] += e;
    }
  };
  for (auto& t : c->timed) add(t);
  if (c->graph_unread && c->last_graph >= 0)
    for (auto& t : c->graphs[c->last_graph].timed) add(t);
  c->graph_unread = false;
  c->recycle_timed();
  return s;
}

const char* lbm_last_error(const lbm_ctx* c) { return c ? c->err.c_str() : "null context"; }

void lbm_destroy(lbm_ctx* c) { delete c; }

}  // extern "C"
