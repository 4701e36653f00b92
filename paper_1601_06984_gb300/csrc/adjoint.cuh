// Discrete adjoint of the multilevel step (reverse mode, hand-written).
//
// Every forward kernel of the path has a reverse here: pull stream + BGK
// collide (Sec. 2.1), the outlet values (Sec. 2.3), the GhostFromCoarser
// source moments and compact interpolation and the GhostFromFiner restriction
// (Sec. 2.2).  A reverse kernel reads the forward state the op saw (from the
// tape) and applies the transposed Jacobian to the adjoint of the op's
// outputs.  The reverse stream-collide stores the adjoint of its inputs, whose
// rows hold nothing yet; the ghosts' adjoints go to compact arrays and are
// added to their sources afterwards.  Scatter targets are unique within one
// launch (each pdf slot is pulled by exactly one element; each ghost has its
// own children; each source element appears once), so plain read-modify-write
// is race-free; the ghost-to-source sums of GhostFromCoarser go through a
// transposed (CSR) list so that they are deterministic too.  Derivatives with
// respect to the relaxation rates and the inlet velocity are summed per block
// into the block's own running row (launches are stream-ordered) and the rows
// are summed once at the end, in block order (deterministic); body-force
// derivatives are accumulated per element in FP64.
#pragma once

#include "kernels.cuh"

namespace lbm {
namespace dev {

// Threads per block.  FP64: small blocks, which spread a small level over all
// SMs (as the forward's kScBlock), two warps rather than one so that the
// block's parameter sums stay a small part of its FP64 work.
template <class S>
constexpr int kAdjBlock = sizeof(typename Sto<S>::R) == 8 ? 64 : 256;
// Minimum resident blocks per SM with 4-byte compute type (FP64: uncapped).
template <class S>
constexpr int adj_minb(int m) { return sizeof(typename Sto<S>::R) == 8 ? 1 : m; }

// ----------------------------------------------------------------- reverse helpers
// Moments M0 = sum P_i, M1_a = sum P_i c_ia, M2_ab = sum P_i c_ia c_ib of
// P_i = w_i lam_i.  The reverse of the equilibrium and of the Guo term is a
// sum over the directions with weights of degree <= 2 in c_i, so it needs
// only these; opposite velocities share them by their sum and difference.
template <int Q, class R>
struct RevSums {
  static constexpr int D = Lat<Q>::D;
  R M0, M1[3], M2[3][3];
  __device__ __forceinline__ explicit RevSums(const R* lam) {
    using LT = Lat<Q>;
    M0 = R(LT::w(0)) * lam[0];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      M1[a] = R(0);
#pragma unroll
      for (int b = 0; b < 3; ++b) M2[a][b] = R(0);
    }
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const R w = R(LT::w(i));
      const R s = w * (lam[i] + lam[i + 1]), d = w * (lam[i] - lam[i + 1]);
      M0 += s;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        if (LT::c(i, a) > 0) M1[a] += d;
        if (LT::c(i, a) < 0) M1[a] -= d;
#pragma unroll
        for (int b = a; b < D; ++b) {
          const int cc = LT::c(i, a) * LT::c(i, b);
          if (cc > 0) M2[a][b] += s;
          if (cc < 0) M2[a][b] -= s;
        }
      }
    }
  }
  // (M2 v)_a
  __device__ __forceinline__ R m2(int a, const R* v) const {
    R s = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) s += (a <= b ? M2[a][b] : M2[b][a]) * v[b];
    return s;
  }
  __device__ __forceinline__ R m1(const R* v) const {
    R s = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) s += M1[a] * v[a];
    return s;
  }
  // reverse of g^eq(rp, rho, u): adds to lam_rp and lam_u
  __device__ __forceinline__ void geq_rev(R rho, const R* u, R usq, R& lam_rp, R* lam_u) const {
    R uM2u = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const R t = m2(a, u);
      uM2u += u[a] * t;
      lam_u[a] += rho * (R(3) * (M1[a] - u[a] * M0) + R(9) * t);
    }
    lam_rp += M0 + R(3) * m1(u) + R(4.5) * uM2u - R(1.5) * usq * M0;
  }
  // reverse of the Guo term (1 - omega/2) w_i [3 (c_i.F - u.F) + 9 (c_i.u)(c_i.F)];
  // without a force only lam_F
  __device__ __forceinline__ void guo_rev(R om, const R* u, const R* F, bool force, R& lam_om, R* lam_u,
                                          R* lam_F) const {
    const R pre = R(1) - R(0.5) * om;
#pragma unroll
    for (int a = 0; a < D; ++a) lam_F[a] += pre * (R(3) * (M1[a] - u[a] * M0) + R(9) * m2(a, u));
    if (!force) return;
    R uF = R(0), uM2F = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const R t = m2(a, F);
      uF += u[a] * F[a];
      uM2F += u[a] * t;
      lam_u[a] += pre * (R(9) * t - R(3) * F[a] * M0);
    }
    lam_om += -R(0.5) * (R(3) * (m1(F) - uF * M0) + R(9) * uM2F);
  }
};

template <int Q, class R>
__device__ __forceinline__ void moments_of(const R* g, R& rp, R* j) {
  if constexpr (sizeof(R) == 8) raw_moments64<Q>(g, rp, j);
  else raw_moments<Q, R>(g, rp, j);
}

// Reverse of post_moments (stored post-collision pdfs -> rp, u, f^neq, S).
// Inputs: the pdfs g, the adjoints of the outputs (lam_fneq is overwritten).
// Outputs: lam_g (assigned), lam_F and lam_om (accumulated).  S_ab = pre sum_i
// c_a c_b f^neq_i with pre = -3 omega / (2 rho), so the adjoint of pre is
// lam_S . S / pre.
template <int Q, class R>
__device__ __forceinline__ void post_moments_rev(const R* g, R om, R rho_off, const R* F, bool force, R lam_rp_in,
                                                 const R* lam_u_in, R* lam_fneq, const R* lam_S, R* lam_g,
                                                 R* lam_F, R& lam_om) {
  using LT = Lat<Q>;
  constexpr int D = LT::D, NS = LT::NS;
  R rp, j[3];
  moments_of<Q, R>(g, rp, j);
  const R rho = rho_off + rp;
  const R inv = R(1) / rho;
  R u[3] = {R(0), R(0), R(0)};
  R usq = R(0);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    u[a] = (force ? j[a] - R(0.5) * F[a] : j[a]) * inv;
    usq += u[a] * u[a];
  }
  const R r1w = R(1) / (R(1) - om);
  const R pre = -R(1.5) * om * inv;
  const R base = rp - R(1.5) * rho * usq;
  // one pair of opposite velocities at a time: f^neq, the strain rate's share
  // of its adjoint, and sum_i lam_fneq_i f^neq_i, sum_ab lam_S_ab S_ab / pre
  R lam_dot = R(0), sdot = R(0);
#pragma unroll
  for (int i = 0; i < Q; i += i ? 2 : 1) {
    R cu = R(0), cF = R(0), uF = R(0), q = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const R c = R(LT::c(i, a));
      if (LT::c(i, a) != 0) {
        cu += c * u[a];
        cF += c * F[a];
      }
      uF += u[a] * F[a];
#pragma unroll
      for (int b = a; b < D; ++b) {
        const int cc = LT::c(i, a) * LT::c(i, b);
        if (cc > 0) q += lam_S[sidx<D>(a, b)];
        if (cc < 0) q -= lam_S[sidx<D>(a, b)];
      }
    }
    const R w = R(LT::w(i));
    R even = w * (base + R(4.5) * rho * cu * cu), odd = w * R(3) * rho * cu;
    if (force) {
      const R fp = (R(1) - R(0.5) * om) * w;
      even += fp * (R(9) * cu * cF - R(3) * uF);
      odd += fp * R(3) * cF;
    }
#pragma unroll
    for (int h = 0; h < (i ? 2 : 1); ++h) {
      const R fn = (g[i + h] - (h ? even - odd : even + odd)) * r1w;
      sdot += q * fn;
      lam_fneq[i + h] += pre * q;
      lam_dot += lam_fneq[i + h] * fn;
    }
  }
  R lam_rho = -pre * sdot * inv;  // d pre / d rho = -pre / rho
  lam_om += -R(1.5) * inv * sdot;
  lam_om += lam_dot * r1w;        // d r1w / d omega = r1w^2
#pragma unroll
  for (int i = 0; i < Q; ++i) lam_g[i] = lam_fneq[i] * r1w;
#pragma unroll
  for (int i = 0; i < Q; ++i) lam_fneq[i] = -lam_g[i];
  const RevSums<Q, R> m(lam_fneq);
  R lam_rp = lam_rp_in;
  R lam_u[3] = {R(0), R(0), R(0)};
#pragma unroll
  for (int a = 0; a < D; ++a) lam_u[a] = lam_u_in[a];
  m.guo_rev(om, u, F, force, lam_om, lam_u, lam_F);
  m.geq_rev(rho, u, usq, lam_rp, lam_u);
  R lam_j[3] = {R(0), R(0), R(0)};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    lam_j[a] = lam_u[a] * inv;
    lam_F[a] += -R(0.5) * lam_j[a];
    lam_rho += -lam_j[a] * u[a];
  }
  lam_rp += lam_rho;
  lam_g[0] += lam_rp;
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    R cl = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (LT::c(i, a) > 0) cl += lam_j[a];
      if (LT::c(i, a) < 0) cl -= lam_j[a];
    }
    lam_g[i] += lam_rp + cl;
    lam_g[i + 1] += lam_rp - cl;
  }
}

// Reverse of one element's BGK collision with Guo forcing (u = (j + F/2) / rho),
// from the pdfs g it pulled and the adjoints lo of its outputs, which become
// the adjoints of the pulled pdfs.  The collision Jacobian is the identity
// times (1 - omega) plus a rank-(1+d) part: with
//   A_i = d g^eq_i / d rp,  B_ia = d g^eq_i / d u_a,  G_ia = d guo_i / d u_a,
//   S0 = sum_i lo_i A_i,   S_a = sum_i lo_i (omega B_ia + G_ia),
// the adjoint of pulled pdf i is
//   (1 - omega) lo_i + base + sum_a c_ia S_a / rho,
//   base = omega S0 - sum_a S_a u_a / rho,
// every sum from RevSums.  lF and lom receive the element's derivatives with
// respect to its force and omega.
template <int Q, class R>
__device__ __forceinline__ void bgk_rev(const R* g, R* lo, const R* F, bool force, R om, R rho_off, R* lF, R& lom) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  R rp, j[3];
  moments_of<Q, R>(g, rp, j);
  const R rho = rho_off + rp, inv = R(1) / rho;
  R u[3] = {R(0), R(0), R(0)}, usq = R(0), uF = R(0);
#pragma unroll
  for (int b = 0; b < D; ++b) {
    u[b] = (force ? j[b] + R(0.5) * F[b] : j[b]) * inv;
    usq += u[b] * u[b];
    uF += u[b] * F[b];
  }
  const R fpre = R(1) - R(0.5) * om;
  R lg_dot = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) lg_dot += lo[i] * g[i];
  const RevSums<Q, R> m(lo);
  R M2u[3] = {R(0), R(0), R(0)}, M2F[3] = {R(0), R(0), R(0)}, uM2u = R(0);
#pragma unroll
  for (int b = 0; b < D; ++b) {
    M2u[b] = m.m2(b, u);
    uM2u += u[b] * M2u[b];
    if (force) M2F[b] = m.m2(b, F);
  }
  // sum lo_i A_i, sum lo_i g^eq_i, sum lo_i Guo_i
  const R quad = R(3) * m.m1(u) + R(4.5) * uM2u - R(1.5) * usq * m.M0;
  lom = rp * m.M0 + rho * quad - lg_dot;
  if (force) {
    R uM2F = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) uM2F += u[b] * M2F[b];
    lom -= R(0.5) * (R(3) * (m.m1(F) - uF * m.M0) + R(9) * uM2F);
  }
  R base = om * (m.M0 + quad), sa[3] = {R(0), R(0), R(0)};
#pragma unroll
  for (int b = 0; b < D; ++b) {
    const R lin = R(3) * (m.M1[b] - u[b] * m.M0) + R(9) * M2u[b];  // sum lo_i B_ib / rho
    R Sa = om * rho * lin;
    if (force) Sa += fpre * (R(9) * M2F[b] - R(3) * F[b] * m.M0);
    sa[b] = Sa * inv;
    lF[b] = fpre * lin + R(0.5) * sa[b];
    base -= sa[b] * u[b];
  }
  const R keep = R(1) - om;
  lo[0] = keep * lo[0] + base;
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    R cs = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      if (LT::c(i, b) > 0) cs += sa[b];
      if (LT::c(i, b) < 0) cs -= sa[b];
    }
    lo[i] = keep * lo[i] + (base + cs);
    lo[i + 1] = keep * lo[i + 1] + (base - cs);
  }
}

// Adds the block's sums to its running row: v[0] to omega of level c.la, v[1]
// to omega of level c.lb, v[2..4] to u_in.  One warp per value sums the
// threads' shares in FP64: NV (threads / 32 + 5) FP64 instructions a block
// (summing in every warp took 4 times as many, on the pipe that is GB300's
// narrowest: 12 us for 1,024 blocks of 256 threads and five values).
template <class R, int NV>
__device__ __forceinline__ void store_partials(const R (&v)[NV], const AdjCommon& c, int row0 = 0) {
  constexpr int MAXT = 256;
  __shared__ R sh[NV][MAXT];
#pragma unroll
  for (int k = 0; k < NV; ++k) sh[k][threadIdx.x] = v[k];
  // the u_in shares only where the block has an inlet link
  int nv = NV;
  if constexpr (NV > 2) {
    if (!__syncthreads_or(v[2] != R(0) || v[3] != R(0) || v[4] != R(0))) nv = 1;
  } else {
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int k = threadIdx.x >> 5; k < nv; k += nw) {
    double s = 0.0;
    for (int t = lane; t < (int)blockDim.x; t += 32) s += (double)sh[k][t];
    s = warp_sum(s);
    if (lane == 0) {
      double* row = c.partial + (size_t)(row0 + blockIdx.x) * kAccCols;
      if (k == 0) row[c.la] += s;
      else if (k == 1) { if (c.lb >= 0) row[c.lb] += s; }
      else row[16 + k - 2] += s;
    }
  }
}

// Read-modify-writes below issue every load before the first store: the
// compiler cannot tell that rows q N + e of one array are distinct, and would
// otherwise wait for each load in turn.
template <class R>
__device__ __forceinline__ void add_force(double* lam_force, int64_t Ntot, int64_t e, const R* lF, int D) {
  if (!lam_force) return;
  double cur[3] = {0.0, 0.0, 0.0};
  for (int b = 0; b < D; ++b) cur[b] = lam_force[(size_t)b * Ntot + e];
  for (int b = 0; b < D; ++b) lam_force[(size_t)b * Ntot + e] = cur[b] + (double)lF[b];
}

// lam[q N + e] += v[q] for q < Q
template <int Q, class R>
__device__ __forceinline__ void add_rows(R* lam, size_t N, int64_t e, const R* v) {
  R cur[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) cur[q] = lam[(size_t)q * N + e];
#pragma unroll
  for (int q = 0; q < Q; ++q) lam[(size_t)q * N + e] = cur[q] + v[q];
}

template <class S, class R>
__device__ __forceinline__ void load_force(const void* force, int64_t Ntot, int64_t e, R* F, int D) {
  F[0] = F[1] = F[2] = R(0);
  if (force)
    for (int b = 0; b < D; ++b) F[b] = static_cast<const R*>(force)[(size_t)b * Ntot + e];
}

// ----------------------------------------------------------------- objective seeds
// Kinetic energy J = sum vol rho |u|^2 / 2 with rho u = j - F/2: dJ/dg_i =
// vol (c_i.u - |u|^2/2), dJ/dF = -vol u / 2.  Obstacle force component k:
// J = sum_links 2 fscale c_opp,k f*_opp  ->  dJ/dg_opp = 2 fscale c_opp,k.
template <int Q, class S>
__global__ void __launch_bounds__(256) k_adj_seed(const AdjSeedArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  const S* __restrict__ x = static_cast<const S*>(a.c.fsrc);
  R* lam = static_cast<R*>(a.c.lam_b);
  const size_t N = (size_t)a.c.Ntot;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a.objective == 0) {
    for (int64_t e = a.begin + t0; e < a.end; e += stride) {
      R g[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) g[q] = Sto<S>::ld(x + (size_t)q * N + e);
      R F[3];
      load_force<S, R>(a.c.force, a.c.Ntot, e, F, D);
      R rp, j[3];
      raw_moments<Q, R>(g, rp, j);
      const R rho = R(a.c.rho_off) + rp;
      R u[3] = {R(0), R(0), R(0)}, usq = R(0);
#pragma unroll
      for (int b = 0; b < D; ++b) {
        u[b] = (j[b] - R(0.5) * F[b]) / rho;
        usq += u[b] * u[b];
      }
      const R vol = R(a.vol);
      R v[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        R cu = R(0);
#pragma unroll
        for (int b = 0; b < D; ++b) cu += R(LT::c(q, b)) * u[b];
        v[q] = vol * (cu - R(0.5) * usq);
      }
      add_rows<Q, R>(lam, N, e, v);
      R lF[3];
#pragma unroll
      for (int b = 0; b < D; ++b) lF[b] = -R(0.5) * vol * u[b];
      add_force<R>(a.c.lam_force, a.c.Ntot, e, lF, D);
    }
  } else {
    // F_k = fscale c_ib,k (f*_ib(x) + f_i(x)), f_i the (interpolated) bounce-
    // back value: pass 0 seeds f*_ib(x), pass 1 f*_ib(x + c_i), pass 2 f*_i(x)
    const int k = a.objective - 1;
    for (int64_t l = t0; l < a.obs_n; l += stride) {
      const int i = a.obs_dir[l];
      const int ib = opp(i);
      const int64_t e = a.obs_elem[l];
      int cb = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (q == ib) cb = LT::c(q, k < D ? k : 0);
      if (k >= D) continue;
      const double q = a.obs_q ? a.obs_q[l] : 0.5;
      const int32_t a2 = a.obs_a ? a.obs_a[l] : -1;
      double w_own, w_a = 0.0, w_i = 0.0;
      if (q < 0.5) {
        w_own = a2 < 0 ? 2.0 : 1.0 + 2.0 * q;
        if (a2 >= 0) w_a = 1.0 - 2.0 * q;
      } else {
        w_own = 1.0 + 1.0 / (2.0 * q);
        w_i = (2.0 * q - 1.0) / (2.0 * q);
      }
      const double base = a.fscale * cb;
      if (a.which == 0) lam[(size_t)ib * N + e] += R(base * w_own);
      if (a.which == 1 && w_a != 0.0) lam[(size_t)ib * N + a2] += R(base * w_a);
      if (a.which == 2 && w_i != 0.0) lam[(size_t)i * N + e] += R(base * w_i);
    }
  }
}

// ----------------------------------------------------------------- stream + collide
// Reverse of the pull + BGK collide.  The pulled pdfs are gathered as the
// forward did (interior bricks, boundary bricks and the neighbour list the
// same way), bgk_rev turns the adjoints of the element's outputs into those
// of the pulled pdfs, and each is stored to the slot the forward pulled from,
// or to the adjoint of the boundary value it came from.  Each slot has one
// reader, and at this point of the reverse sweep its adjoint holds nothing
// yet: the state the step read has no later reader, and the fills and moments
// before the step add to it afterwards.  So the streaming is a plain store
// (no read-modify-write), and an interior brick's own output adjoints need
// not be cleared: all their slots are stored again by the step before, whose
// readers are all there.  The other elements' are cleared, since some of their
// slots have no reader (beside ghosts that are not advanced, at an outlet).
// Bound by L2 and latency: 19 + 19 loads and 19 (interior) or 38 stores per
// element; 57 and 38 with the read-modify-write.  FP32, 64^3 two-level flow,
// mean of its launches: interior 23.4 -> 19.2 us, the rest beside it (all list
// elements then, three quarters of them boundary bricks now) 37.7 -> 16.4 us.
template <int Q, class S>
__global__ void __launch_bounds__(kAdjBlock<S>, adj_minb<S>(3)) k_adj_sc_interior(const __grid_constant__ AdjSCArgs a) {
  using R = typename Sto<S>::R;
  constexpr int D = Lat<Q>::D;
  const int64_t t = (int64_t)blockIdx.x * kAdjBlock<S> + threadIdx.x;
  const int l = (int)t & 63, lane = threadIdx.x & 31;
  // the brick index is uniform over each warp, so the shuffles run with whole warps
  const int64_t b = t >> 6;
  R part[1] = {R(0)};
  if (b < a.n_interior) {
    BrickLinks<Q> k;
    k.load(a.brick_tab, a.brick_nb, b, l, lane);
    const size_t N = (size_t)a.c.Ntot;
    const int64_t first = a.begin + b * 64, e = first + l;
    const S* __restrict__ x = static_cast<const S*>(a.c.fsrc) + first;
    const R* __restrict__ lam_out = static_cast<const R*>(a.c.lam_a) + e;
    R* __restrict__ lam_in = static_cast<R*>(a.c.lam_b) + first;
    // pull source of link i: row i of the state, at this 32-bit offset from
    // the brick's first element (kept, not the 64-bit addresses)
    int32_t off[Q];
    off[0] = l;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const uint32_t v = k.entry(i);
      off[i] = __shfl_sync(0xffffffffu, k.row, (int)(v >> 6)) + (int32_t)(v & 63);
    }
    R g[Q], lo[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = Sto<S>::ld(x + (int64_t)(i * N) + off[i]);
#pragma unroll
    for (int i = 0; i < Q; ++i) lo[i] = lam_out[(size_t)i * N];
    R F[3], lF[3];
    load_force<S, R>(a.c.force, a.c.Ntot, e, F, D);
    bgk_rev<Q, R>(g, lo, F, a.c.force != nullptr, R(a.omega), R(a.c.rho_off), lF, part[0]);
    add_force<R>(a.c.lam_force, a.c.Ntot, e, lF, D);
#pragma unroll
    for (int i = 0; i < Q; ++i) lam_in[(int64_t)(i * N) + off[i]] = lo[i];
  }
  store_partials<R, 1>(part, a.c);
}

// Boundary bricks (the first blocks) and the elements of the neighbour-list
// range, links resolved as in k_sc_rest.
template <int Q, class S>
__global__ void __launch_bounds__(kAdjBlock<S>, adj_minb<S>(2)) k_adj_sc_rest(const __grid_constant__ AdjSCArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  const size_t N = (size_t)a.c.Ntot;
  R part[5] = {R(0), R(0), R(0), R(0), R(0)};
  const int64_t t = (int64_t)blockIdx.x * kAdjBlock<S> + threadIdx.x;
  const bool list = (int)blockIdx.x >= a.bnd_blocks;  // uniform over the block
  int32_t off[Q];
  uint32_t miss = 0;
  int64_t first = 0;
  int l = 0;
  bool active;
  if (list) {
    const int64_t lin = a.list_begin + (t - (int64_t)a.bnd_blocks * kAdjBlock<S>);
    active = lin < a.list_end;
    if (active) {
      first = lin + (lin >= a.hole_at ? a.hole_len : 0);
#pragma unroll
      for (int i = 1; i < Q; ++i) off[i] = (int32_t)__ldg(a.nbr + (size_t)(i - 1) * N + first);
      miss = ~0u;
    }
  } else {
    const int64_t b = t >> 6;  // uniform over the warp
    active = b < a.n_boundary;
    if (active) {
      l = (int)t & 63;
      BrickLinks<Q> k;
      k.load(a.brick_tab, a.brick_nb + (size_t)a.n_interior * 27, b, l, threadIdx.x & 31);
      first = a.begin + (a.n_interior + b) * 64;
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const uint32_t v = k.entry(i);
        const int32_t r = __shfl_sync(0xffffffffu, k.row, (int)(v >> 6));
        if (r != kBrickMissing) {
          off[i] = r + (int32_t)(v & 63);
        } else {
          off[i] = (int32_t)__ldg(a.nbr + (size_t)(i - 1) * N + first + l);
          miss |= 1u << i;
        }
      }
    }
  }
  if (active) {
    uint32_t patch = 0;  // links with an inlet term or a boundary value
    off[0] = l;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if (!((miss >> i) & 1u)) continue;
      const uint32_t n = (uint32_t)off[i];
      if (n < NB_FLAG30) {
        off[i] = (int32_t)((int64_t)n - first);
      } else {
        off[i] = (int32_t)((int64_t)(opp(i) - i) * (int64_t)N + l);
        if (n & NB_FLAG30) patch |= 1u << i;
      }
    }
    const int64_t e = first + l;
    const S* __restrict__ x = static_cast<const S*>(a.c.fsrc) + first;
    R* __restrict__ lam_out = static_cast<R*>(a.c.lam_a) + e;
    R* __restrict__ lam_in = static_cast<R*>(a.c.lam_b) + first;
    R g[Q], lo[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = Sto<S>::ld(x + (int64_t)(i * N) + off[i]);
#pragma unroll
    for (int i = 0; i < Q; ++i) lo[i] = lam_out[(size_t)i * N];
    const auto code = [&](int i) { return __ldg(a.nbr + (size_t)(i - 1) * N + e); };
    const auto profile = [&](uint32_t n) { return a.inlet_s ? R(a.inlet_s[n & NB_INDEX]) : R(1); };
    if (patch) {
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        if (!((patch >> i) & 1u)) continue;
        const uint32_t n = code(i);
        if (n & NB_BOUNCE) g[i] += R(a.inlet[i]) * profile(n);
        else g[i] = static_cast<const R*>(a.side_fwd)[n & NB_INDEX];
      }
    }
    R F[3], lF[3];
    load_force<S, R>(a.c.force, a.c.Ntot, e, F, D);
    bgk_rev<Q, R>(g, lo, F, a.c.force != nullptr, R(a.omega), R(a.c.rho_off), lF, part[0]);
    add_force<R>(a.c.lam_force, a.c.Ntot, e, lF, D);
    if (!patch) {
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        lam_out[(size_t)i * N] = R(0);
        lam_in[(int64_t)(i * N) + off[i]] = lo[i];
      }
    } else {
      lam_out[0] = R(0);
      lam_in[off[0]] = lo[0];
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        lam_out[(size_t)i * N] = R(0);
        const bool special = (patch >> i) & 1u;
        const uint32_t n = special ? code(i) : 0u;
        if (special && !(n & NB_BOUNCE)) {
          static_cast<R*>(a.lam_side)[n & NB_INDEX] = lo[i];
          continue;
        }
        lam_in[(int64_t)(i * N) + off[i]] = lo[i];
        if (special) {
          // d f_i / d u_in = 6 w_i rho0 s c_i, s the link's inlet profile factor
          const R sf = profile(n);
#pragma unroll
          for (int b = 0; b < D; ++b) part[2 + b] += lo[i] * sf * R(6.0 * LT::w(i) * a.c.rho0 * LT::c(i, b));
        }
      }
    }
  }
  store_partials<R, 5>(part, a.c, a.row0);
}

// ----------------------------------------------------------------- outlet values
template <int Q, class S>
__global__ void __launch_bounds__(256) k_adj_outlet(const AdjOutletArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  constexpr int D = LT::D, NS = LT::NS;
  const S* __restrict__ x = static_cast<const S*>(a.c.fsrc);
  R* lam_in = static_cast<R*>(a.c.lam_b);
  const R* lam_side = static_cast<const R*>(a.lam_side);
  const size_t N = (size_t)a.c.Ntot;
  R part[1] = {R(0)};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = a.begin + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.end; k += stride) {
    const int i = a.dir[k];
    const R ls = lam_side[k];
    if (a.kind[k] == OUT_EXTRAP) {
      if (a.which == 1) lam_in[(size_t)i * N + a.a[k]] += a.zero_gradient ? ls : R(2) * ls;
      if (a.which == 2 && !a.zero_gradient) lam_in[(size_t)i * N + a.b[k]] -= ls;
      continue;
    }
    if (a.kind[k] == OUT_BOUZIDI) {
      // interpolated bounce-back value, linear in f*_i(x) (pass 3), f*_ib(x)
      // (pass 4) and f*_ib(x + c_i) (pass 5); one slot per link and pass
      const int ib = opp(i);
      const int64_t e = a.elem[k];
      const double q = a.q ? a.q[k] : 0.5;
      const int32_t a2 = a.a[k];
      if (q < 0.5) {
        if (a.which == 4) lam_in[(size_t)ib * N + e] += a2 < 0 ? ls : R(2.0 * q) * ls;
        if (a.which == 5 && a2 >= 0) lam_in[(size_t)ib * N + a2] += R(1.0 - 2.0 * q) * ls;
      } else {
        if (a.which == 4) lam_in[(size_t)ib * N + e] += R(1.0 / (2.0 * q)) * ls;
        if (a.which == 3) lam_in[(size_t)i * N + e] += R((2.0 * q - 1.0) / (2.0 * q)) * ls;
      }
      continue;
    }
    if (a.which != 0) continue;
    // side = g^eq_i(rho0, u) + f^neq_ib, with u and the pre-collision f^neq
    // taken from the stored pdfs g (post_moments)
    const int64_t e = a.elem[k];
    R g[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) g[q] = Sto<S>::ld(x + (size_t)q * N + e);
    R F[3];
    load_force<S, R>(a.c.force, a.c.Ntot, e, F, D);
    R rp, j[3];
    raw_moments<Q, R>(g, rp, j);
    const R rho = R(a.c.rho_off) + rp, inv = R(1) / rho;
    R u[3] = {R(0), R(0), R(0)}, usq = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      u[b] = (j[b] - R(0.5) * F[b]) * inv;
      usq += u[b] * u[b];
    }
    const int ib = opp(i);
    // term g^eq_i(rho0, u): depends on u only
    R lam_rp_dummy = R(0), lam_u[3] = {R(0), R(0), R(0)};
    R l1[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) l1[q] = q == i ? ls : R(0);
    RevSums<Q, R>(l1).geq_rev(R(a.c.rho0), u, usq, lam_rp_dummy, lam_u);
    // term f^neq_ib, and u's dependence on g
    R lfn[Q], lS[NS], lg[Q], lF[3] = {R(0), R(0), R(0)}, lom = R(0);
#pragma unroll
    for (int q = 0; q < Q; ++q) lfn[q] = q == ib ? ls : R(0);
#pragma unroll
    for (int s2 = 0; s2 < NS; ++s2) lS[s2] = R(0);
    post_moments_rev<Q, R>(g, R(a.omega), R(a.c.rho_off), F, a.c.force != nullptr, R(0), lam_u, lfn, lS, lg, lF, lom);
    add_rows<Q, R>(lam_in, N, e, lg);
    add_force<R>(a.c.lam_force, a.c.Ntot, e, lF, D);
    part[0] += lom;
  }
  if (a.which == 0) store_partials<R, 1>(part, a.c);
}

// ----------------------------------------------------------------- source moments
// Coefficients of a ghost's local-frame velocity adjoint L in the adjoints of
// the strain-rate differences of its four sources (the transpose of
// compact_uloc): aD[x][c] for the difference D_x of component c.
template <int Q, class R>
__device__ __forceinline__ void compact_rev(const R* L, R (&aD)[3][Lat<Q>::NS]) {
  constexpr int D = Lat<Q>::D, NS = Lat<Q>::NS;
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int c = 0; c < NS; ++c) aD[x][c] = R(0);
  if constexpr (D == 3) {
    constexpr int XX = 0, YY = 1, ZZ = 2, XY = 3, YZ = 4, XZ = 5;
    const R p0 = R(-0.1875) * L[0], p1 = R(-0.1875) * L[1], p2 = R(-0.1875) * L[2];
    const R r0 = R(-0.0625) * L[0], r1 = R(-0.0625) * L[1], r2 = R(-0.0625) * L[2], r = r0 + r1 + r2;
    aD[0][XX] = R(0.5) * p0, aD[0][YY] = r1 - R(0.5) * p0, aD[0][ZZ] = r2 - R(0.5) * p0;
    aD[0][XY] = p1, aD[0][XZ] = p2, aD[0][YZ] = r - R(2) * r0;
    aD[1][XX] = r0 - R(0.5) * p1, aD[1][YY] = R(0.5) * p1, aD[1][ZZ] = r2 - R(0.5) * p1;
    aD[1][XY] = p0, aD[1][YZ] = p2, aD[1][XZ] = r - R(2) * r1;
    aD[2][XX] = r0 - R(0.5) * p2, aD[2][YY] = r1 - R(0.5) * p2, aD[2][ZZ] = R(0.5) * p2;
    aD[2][XZ] = p0, aD[2][YZ] = p1, aD[2][XY] = r - R(2) * r2;
  } else {
    const R p0 = R(-0.1875) * L[0], p1 = R(-0.1875) * L[1], r0 = R(0.0625) * L[0], r1 = R(0.0625) * L[1];
    aD[0][0] = R(0.5) * p0, aD[0][1] = r1 - R(0.5) * p0, aD[0][2] = p1;
    aD[1][0] = r0 - R(0.5) * p1, aD[1][1] = R(0.5) * p1, aD[1][2] = p0;
  }
}

// Values k_adj_gfc leaves per ghost: the scaled adjoints of its f^neq
// (padded to a multiple of 4), then of its density and its local-frame velocity.
template <int Q>
constexpr int kGhostAdj = (Q + 3) / 4 * 4 + 4;

// Reverse of the source records, one thread per source (64^3 two-level flow,
// FP32: 12.5 us; the sum over four records' adjoints per ghost and the reverse
// of the records as two kernels took 17.3 + 9.8 us): sums what its ghosts
// leave for it (k_adj_gfc; fixed order: the transposed list), which is the
// adjoint of its record, and takes it back to the source's pdfs.  LINEAR mode:
// the record at t + 1/2 is the mean of those at t and t + 1; its reverse (half
// set) applies half to the state at t + 1 and leaves half in rec_half, which
// the reverse of the fill at t adds (rec_half without half).
// LANES consecutive lanes share a source's ghosts (about ten items, each a
// chain of two loads), four where the sources alone would not fill the GPU:
// 64^3 FP32 15.7 -> 12.5 us, D2Q9 FP64 with 450 sources 26 -> 17 us.
template <int Q, class S, int LANES>
__global__ void __launch_bounds__(sizeof(typename Sto<S>::R) == 8 ? 32 : 128) k_adj_moments(const __grid_constant__ AdjMomArgs a) {
  using R = typename Sto<S>::R;
  using RL = RecLayout<Q>;
  constexpr int D = Lat<Q>::D, NS = Lat<Q>::NS, CS = kGhostAdj<Q>;
  const S* __restrict__ x = static_cast<const S*>(a.c.fsrc);
  R* lam_in = static_cast<R*>(a.c.lam_b);
  const R* __restrict__ ghosts = static_cast<const R*>(a.contrib);
  const size_t N = (size_t)a.c.Ntot;
  R part[1] = {R(0)};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // whole warps iterate together (the shuffles below)
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t - threadIdx.x % 32 < a.nsrc * LANES; t += stride) {
    const int64_t k = t / LANES;
    const bool active = k < a.nsrc;
    R lfn[Q], lS[NS], lu[3] = {R(0), R(0), R(0)}, lrp = R(0);
#pragma unroll
    for (int q = 0; q < Q; ++q) lfn[q] = R(0);
#pragma unroll
    for (int s = 0; s < NS; ++s) lS[s] = R(0);
    const int j1 = active ? a.off[k + 1] : 0;
    for (int j = active ? a.off[k] + (int)(t % LANES) : 0; j < j1; j += LANES) {
      const int item = a.item[j], slot = item & 3, oct = (item >> 2) & ((1 << D) - 1);
      const R* __restrict__ v = ghosts + (size_t)(item >> 2) * CS;
      R h[CS];
#pragma unroll
      for (int f = 0; f < CS; f += 4) ld4(v + f, h + f);
      const R* L = h + CS - 3;
      // linear weights of density and f^neq, of the velocity, and the signs of
      // the source's strain rate in the differences
      const R lw = D == 3 ? (slot == 0 ? R(0.625) : R(0.125))
                          : (slot == 0 ? R(0.5625) : slot == 3 ? R(0.0625) : R(0.1875));
      const R uw = D == 3 ? lw : (slot == 0 ? R(0.5) : slot == 3 ? R(0) : R(0.25));
      const int neg[3] = {D == 3 ? (0x9 >> slot) & 1 : (0x5 >> slot) & 1,
                          D == 3 ? (0x5 >> slot) & 1 : (0x3 >> slot) & 1, (0x3 >> slot) & 1};
#pragma unroll
      for (int q = 0; q < Q; ++q) lfn[q] += lw * h[q];
      lrp += lw * h[CS - 4];
      R aD[3][NS];
      compact_rev<Q, R>(L, aD);
#pragma unroll
      for (int b = 0; b < D; ++b) {
        lu[b] += ((oct >> b) & 1 ? uw : -uw) * L[b];
#pragma unroll
        for (int c = b; c < D; ++c) {
          const int s = sidx<D>(b, c);
          R t = R(0);
#pragma unroll
          for (int y = 0; y < D; ++y) t += neg[y] ? -aD[y][s] : aD[y][s];
          lS[s] += (b != c && (((oct >> b) ^ (oct >> c)) & 1)) ? R(-0.5) * t : R(0.5) * t;
        }
      }
    }
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1) {
#pragma unroll
      for (int q = 0; q < Q; ++q) lfn[q] += __shfl_xor_sync(0xffffffffu, lfn[q], o);
      lrp += __shfl_xor_sync(0xffffffffu, lrp, o);
#pragma unroll
      for (int b = 0; b < D; ++b) lu[b] += __shfl_xor_sync(0xffffffffu, lu[b], o);
#pragma unroll
      for (int s = 0; s < NS; ++s) lS[s] += __shfl_xor_sync(0xffffffffu, lS[s], o);
    }
    if (!active || t % LANES != 0) continue;
    if (a.rec_half) {
      R* __restrict__ half = static_cast<R*>(a.rec_half) + (size_t)k * RL::STRIDE;
      R rec[RL::STRIDE];
      if (a.half) {
#pragma unroll
        for (int f = 0; f < RL::STRIDE; ++f) rec[f] = R(0);
#pragma unroll
        for (int q = 0; q < Q; ++q) rec[RL::FN + q] = lfn[q] *= R(0.5);
        rec[RL::RP] = lrp *= R(0.5);
#pragma unroll
        for (int b = 0; b < D; ++b) rec[RL::U + b] = lu[b] *= R(0.5);
#pragma unroll
        for (int s = 0; s < NS; ++s) rec[RL::SS + s] = lS[s] *= R(0.5);
#pragma unroll
        for (int f = 0; f < RL::END; f += 4) st4(half + f, rec + f);
      } else {
#pragma unroll
        for (int f = 0; f < RL::END; f += 4) ld4(half + f, rec + f);
#pragma unroll
        for (int q = 0; q < Q; ++q) lfn[q] += rec[RL::FN + q];
        lrp += rec[RL::RP];
#pragma unroll
        for (int b = 0; b < D; ++b) lu[b] += rec[RL::U + b];
#pragma unroll
        for (int s = 0; s < NS; ++s) lS[s] += rec[RL::SS + s];
      }
    }
    const int64_t e = a.elem[k];
    R g[Q];
    load_source<Q, S>(a.saved, x, N, e, k, g);
    R F[3];
    load_force<S, R>(a.c.force, a.c.Ntot, e, F, D);
    R lg[Q], lF[3] = {R(0), R(0), R(0)}, lom = R(0);
    post_moments_rev<Q, R>(g, R(a.omega), R(a.c.rho_off), F, a.c.force != nullptr, lrp, lu, lfn, lS, lg, lF, lom);
    add_rows<Q, R>(lam_in, N, e, lg);
    add_force<R>(a.c.lam_force, a.c.Ntot, e, lF, D);
    part[0] += lom;
  }
  store_partials<R, 1>(part, a.c);
}

// ----------------------------------------------------------------- GhostFromCoarser
// Reverse of the fill up to the sources' records, one thread per ghost: its
// adjoints (cleared) become those of its interpolated f^neq, density and
// local-frame velocity, kGhostAdj values instead of the adjoints of four
// records (96 against 512 bytes a ghost; 52,288 ghosts 25.5 -> 12.2 us), from
// which k_adj_moments forms each source's share.
template <int Q, class S>
__global__ void __launch_bounds__(sizeof(typename Sto<S>::R) == 8 ? 32 : 128) k_adj_gfc(const __grid_constant__ AdjGfcArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  using RL = RecLayout<Q>;
  constexpr int D = LT::D, NS = LT::NS, CS = kGhostAdj<Q>;
  R* __restrict__ lam = static_cast<R*>(a.c.lam_a);
  const R* __restrict__ mom = static_cast<const R*>(a.rec);
  const size_t N = (size_t)a.c.Ntot;
  R part[2] = {R(0), R(0)};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.ng; k += stride) {
    const R* rec[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) rec[s] = mom + (size_t)a.gsrc[(size_t)s * a.ng + k] * RL::STRIDE;
    const uint8_t oct = a.oct[k];
    R sg[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) sg[b] = ((oct >> b) & 1) ? R(1) : R(-1);
    R ul[4][3], Sl[4][NS], rps[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      ul[s][0] = ul[s][1] = ul[s][2] = R(0);
      rps[s] = rec[s][RL::RP];
#pragma unroll
      for (int b = 0; b < D; ++b) ul[s][b] = sg[b] * rec[s][RL::U + b];
#pragma unroll
      for (int b = 0; b < D; ++b)
#pragma unroll
        for (int c = b; c < D; ++c) Sl[s][sidx<D>(b, c)] = sg[b] * sg[c] * rec[s][RL::SS + sidx<D>(b, c)];
    }
    R uloc[3];
    compact_uloc<Q, R>(ul, Sl, uloc);
    R u[3] = {R(0), R(0), R(0)}, usq = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      u[b] = sg[b] * uloc[b];
      usq += u[b] * u[b];
    }
    const R lw[4] = {D == 3 ? R(0.625) : R(0.5625), D == 3 ? R(0.125) : R(0.1875), D == 3 ? R(0.125) : R(0.1875),
                     D == 3 ? R(0.125) : R(0.0625)};
    const R rp = lw[0] * rps[0] + lw[1] * rps[1] + lw[2] * rps[2] + lw[3] * rps[3];
    const R rho = R(a.c.rho_off) + rp;
    const R wf = R(a.omega_f), wc = R(a.omega_c);
    const R scale = (R(1) - wf) * wc / (R(2) * wf);
    const int64_t e = a.dest0 + k;
    // all loads before the ghost's adjoint is zeroed, so that they overlap
    R lo[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) lo[q] = lam[(size_t)q * N + e];
    R lam_scale = R(0);
#pragma unroll
    for (int q0 = 0; q0 < Q; q0 += 4) {
      R f[4][4];
#pragma unroll
      for (int s = 0; s < 4; ++s) ld4(rec[s] + RL::FN + q0, f[s]);
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (q0 + t < Q) lam_scale += lo[q0 + t] * (lw[0] * f[0][t] + lw[1] * f[1][t] + lw[2] * f[2][t] + lw[3] * f[3][t]);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) lam[(size_t)q * N + e] = R(0);
    part[0] += lam_scale * (R(1) - wf) / (R(2) * wf);  // d scale / d omega_c
    part[1] += lam_scale * (-wc / (R(2) * wf * wf));    // d scale / d omega_f
    R lam_rp = R(0), lam_u[3] = {R(0), R(0), R(0)};
    RevSums<Q, R>(lo).geq_rev(rho, u, usq, lam_rp, lam_u);
    R* __restrict__ out = static_cast<R*>(a.contrib) + (size_t)k * CS;
    R v[CS];
#pragma unroll
    for (int f = 0; f < CS; ++f) v[f] = R(0);
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = scale * lo[q];
    v[CS - 4] = lam_rp;
#pragma unroll
    for (int b = 0; b < D; ++b) v[CS - 3 + b] = sg[b] * lam_u[b];
#pragma unroll
    for (int f = 0; f < CS; f += 4) st4(out + f, v + f);
  }
  store_partials<R, 2>(part, a.c);
}

// ----------------------------------------------------------------- GhostFromFiner
// One group of 2^d consecutive lanes per ghost, lane b its child b, as in the
// forward fill: the ghost's density and velocity are sums of d + 1 shares of
// its children over the group, and every lane takes the ghost's adjoints back
// to its own child.  The f^neq sum enters only through the derivative of its
// factor, sum_q lam_q sum_children f^neq_q, of which every lane adds its
// child's part.  (Shuffling the children's f^neq and strain rates too took 41
// values through three steps: 29.3 us for 10,816 ghosts, 16.1 us now.)
template <int Q, class S>
__global__ void __launch_bounds__(kAdjBlock<S>, adj_minb<S>(2)) k_adj_gff(const __grid_constant__ AdjGffArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  constexpr int D = LT::D, NS = LT::NS, NCH = 1 << D;
  const S* __restrict__ x = static_cast<const S*>(a.c.fsrc);
  // coarse ghosts and fine children: disjoint slots, possibly of one buffer
  R* __restrict__ lam_c = static_cast<R*>(a.c.lam_a);
  R* __restrict__ lam_f = static_cast<R*>(a.c.lam_b);
  const size_t N = (size_t)a.c.Ntot;
  const R wf = R(a.omega_f), wc = R(a.omega_c), rho_off = R(a.c.rho_off);
  const bool force = a.c.force != nullptr;
  const R r1w = R(1) / (R(1) - wf);
  R part[2] = {R(0), R(0)};
  const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
  // every lane of a warp runs the same number of iterations (the shuffles need the whole warp)
  const int64_t total = (a.ng * NCH + 31) / 32 * 32;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t - threadIdx.x % 32 < total; t += gstride) {
    const int64_t k = t / NCH;
    const int b = (int)(t % NCH);
    const bool active = k < a.ng;
    R g[Q], F[3] = {R(0), R(0), R(0)};
    R rp = R(0), u[3] = {R(0), R(0), R(0)}, fneq[Q], Sv[NS], lo[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) g[q] = fneq[q] = lo[q] = R(0);
#pragma unroll
    for (int s = 0; s < NS; ++s) Sv[s] = R(0);
    int64_t ec = 0, eg = 0;
    if (active) {
      ec = (int64_t)a.child0[k] + b;
      eg = k < a.n_inner ? a.dest0 + k : a.dest_outer + (k - a.n_inner);
#pragma unroll
      for (int q = 0; q < Q; ++q) g[q] = Sto<S>::ld(x + (size_t)q * N + ec);
#pragma unroll
      for (int q = 0; q < Q; ++q) lo[q] = lam_c[(size_t)q * N + eg];
      load_force<S, R>(a.c.force, a.c.Ntot, ec, F, D);
      if (force) post_moments<Q, R, true, true>(g, wf, r1w, rho_off, F, rp, u, fneq, Sv);
      else post_moments<Q, R, true, false>(g, wf, r1w, rho_off, F, rp, u, fneq, Sv);
    }
    const R inv = R(1) / R(NCH);
    const R lapc = R(2) * R(D == 3 ? 0.5 : 1.0) / R(32);  // dt ratio x difference factor / 32
    R tr = R(0);
#pragma unroll
    for (int c = 0; c < D; ++c) tr += Sv[c];
    R rpm = rp * inv, uP[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int aa = 0; aa < D; ++aa) {
      R s2 = R(0);
#pragma unroll
      for (int c = 0; c < D; ++c) s2 += (b >> c) & 1 ? Sv[sidx<D>(aa, c)] : -Sv[sidx<D>(aa, c)];
      uP[aa] = u[aa] * inv - lapc * (R(2) * s2 - ((b >> aa) & 1 ? tr : -tr));
    }
#pragma unroll
    for (int o = 1; o < NCH; o <<= 1) {
      rpm += __shfl_xor_sync(0xffffffffu, rpm, o);
#pragma unroll
      for (int c = 0; c < D; ++c) uP[c] += __shfl_xor_sync(0xffffffffu, uP[c], o);
    }
    // every lane of the group reads all of the ghost's adjoints, and each
    // clears its share of them: the shuffles order no memory accesses, so the
    // warp waits here, inactive lanes too
    __syncwarp();
    if (!active) continue;
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (q % NCH == b) lam_c[(size_t)q * N + eg] = R(0);
    R usq = R(0);
#pragma unroll
    for (int aa = 0; aa < D; ++aa) usq += uP[aa] * uP[aa];
    const R rho = rho_off + rpm;
    const R scale = (R(1) - wc) * R(2) * wf / wc * inv;
    R lam_scale = R(0);
#pragma unroll
    for (int q = 0; q < Q; ++q) lam_scale += lo[q] * fneq[q];
    part[0] += lam_scale * (R(2) * wf * inv) * (-R(1) / (wc * wc));  // d scale / d omega_c
    part[1] += lam_scale * (R(1) - wc) * R(2) / wc * inv;            // d scale / d omega_f
    R lam_rpm = R(0), lam_uP[3] = {R(0), R(0), R(0)};
    RevSums<Q, R>(lo).geq_rev(rho, uP, usq, lam_rpm, lam_uP);
    // this lane's child
    R lS[NS], lu[3] = {R(0), R(0), R(0)}, lfn[Q];
#pragma unroll
    for (int s = 0; s < NS; ++s) lS[s] = R(0);
#pragma unroll
    for (int aa = 0; aa < D; ++aa) {
      const R ll = -lapc * lam_uP[aa];
      lu[aa] = lam_uP[aa] * inv;
#pragma unroll
      for (int c = 0; c < D; ++c) {
        lS[sidx<D>(aa, c)] += (b >> c) & 1 ? R(2) * ll : R(-2) * ll;
        lS[c] -= (b >> aa) & 1 ? ll : -ll;
      }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) lfn[q] = scale * lo[q];
    R lg[Q], lF[3] = {R(0), R(0), R(0)}, lom = R(0);
    post_moments_rev<Q, R>(g, wf, rho_off, F, force, lam_rpm * inv, lu, lfn, lS, lg, lF, lom);
    add_rows<Q, R>(lam_f, N, ec, lg);
    add_force<R>(a.c.lam_force, a.c.Ntot, ec, lF, D);
    part[1] += lom;
  }
  store_partials<R, 2>(part, a.c);
}

// ----------------------------------------------------------------- launchers
template <class S>
struct AdjLaunch {
  static void seed(int Q, const AdjSeedArgs& a, cudaStream_t st) {
    const int64_t n = a.objective == 0 ? a.end - a.begin : a.obs_n;
    with_q(Q, [&](auto q) { k_adj_seed<decltype(q)::value, S><<<adj_grid(n, 256), 256, 0, st>>>(a); });
  }
  static void sc_interior(int Q, const AdjSCArgs& a, cudaStream_t st) {
    if (a.n_interior <= 0) return;
    with_q(Q, [&](auto q) {
      k_adj_sc_interior<decltype(q)::value, S><<<blocks_for(64 * a.n_interior, kAdjBlock<S>), kAdjBlock<S>, 0, st>>>(a);
    });
  }
  static void sc_rest(int Q, AdjSCArgs& a, cudaStream_t st) {
    a.bnd_blocks = (int)blocks_for(64 * a.n_boundary, kAdjBlock<S>);
    const unsigned g = a.bnd_blocks + (a.list_end > a.list_begin ? blocks_for(a.list_end - a.list_begin, kAdjBlock<S>) : 0);
    if (!g) return;
    with_q(Q, [&](auto q) { k_adj_sc_rest<decltype(q)::value, S><<<g, kAdjBlock<S>, 0, st>>>(a); });
  }
  static void outlet(int Q, const AdjOutletArgs& a, cudaStream_t st) {
    if (a.end <= a.begin) return;
    with_q(Q, [&](auto q) {
      k_adj_outlet<decltype(q)::value, S><<<adj_grid(a.end - a.begin, kAdjLinkBlock), kAdjLinkBlock, 0, st>>>(a);
    });
  }
  static constexpr int kGhostBlock = sizeof(typename Sto<S>::R) == 8 ? 32 : 128;
  static void moments(int Q, const AdjMomArgs& a, cudaStream_t st) {
    if (a.nsrc <= 0) return;
    // four lanes a source up to a warp per SM (FP64, where the extra lanes are
    // extra FP64 instructions) or four blocks per SM
    const bool four = a.nsrc <= (kGhostBlock == 32 ? 152 * 32 : 152 * 4 * 128);
    with_q(Q, [&](auto q) {
      constexpr int QQ = decltype(q)::value;
      if (four) k_adj_moments<QQ, S, 4><<<adj_grid(4 * a.nsrc, kGhostBlock), kGhostBlock, 0, st>>>(a);
      else k_adj_moments<QQ, S, 1><<<adj_grid(a.nsrc, kGhostBlock), kGhostBlock, 0, st>>>(a);
    });
  }
  static void gfc(int Q, const AdjGfcArgs& a, cudaStream_t st) {
    if (a.ng <= 0) return;
    with_q(Q, [&](auto q) {
      k_adj_gfc<decltype(q)::value, S><<<adj_grid(a.ng, kGhostBlock), kGhostBlock, 0, st>>>(a);
    });
  }
  static void gff(int Q, const AdjGffArgs& a, cudaStream_t st) {
    if (a.ng <= 0) return;
    with_q(Q, [&](auto q) {
      constexpr int QQ = decltype(q)::value;
      k_adj_gff<QQ, S><<<adj_grid(a.ng << Lat<QQ>::D, kAdjBlock<S>), kAdjBlock<S>, 0, st>>>(a);
    });
  }
};

template <class S>
const AdjOps* make_adj_ops() {
  static const AdjOps ops = {&AdjLaunch<S>::seed,    &AdjLaunch<S>::sc_interior, &AdjLaunch<S>::sc_rest,
                             &AdjLaunch<S>::outlet,  &AdjLaunch<S>::moments, &AdjLaunch<S>::gfc,
                             &AdjLaunch<S>::gff,     sizeof(typename Sto<S>::R), kAdjBlock<S>, AdjLaunch<S>::kGhostBlock};
  return &ops;
}

}  // namespace dev
}  // namespace lbm
