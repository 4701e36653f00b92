// Device kernels of the multilevel lattice Boltzmann hot path (sm_103a).
//
// Storage S is double (LBM_FP64), float or bfloat16 (deviation storage
// g_i = f_i - w_i rho0, arithmetic in float).  Every kernel is written in the
// deviation form with an offset rho_off (0 for FP64, rho0 otherwise):
//   rho = rho_off + sum g,  g^eq_i = w_i [ (rho - rho_off) + rho (3 c.u + 9/2 (c.u)^2 - 3/2 u.u) ],
// which is Eq. (feq) of Sec. 2.1 minus w_i rho_off.
//
// Memory layout: pdfs A, B as [Q][Ntot] structure-of-arrays over all levels
// (each level a contiguous, padded index range); pull neighbour indices
// nbr[Q-1][Ntot] (uint32, see lbm_internal.h).  One thread per element; the
// direction loops are fully unrolled so every load/store of a warp touches 32
// consecutive elements of one direction array (coalesced), except the pull
// gathers, whose locality comes from the z-curve order.
#pragma once

#include <cuda_bf16.h>
#include <algorithm>
#include <type_traits>
#include <cuda_runtime.h>

#include "lbm_internal.h"

namespace lbm {
namespace dev {

// ----------------------------------------------------------------- lattices
template <int Q>
struct Lat;

template <>
struct Lat<9> {
  static constexpr int D = 2, NS = 3;
  __host__ __device__ static constexpr int c(int i, int a) {
    return a == 0   ? ((i == 1 || i == 5 || i == 7) ? 1 : (i == 2 || i == 6 || i == 8) ? -1 : 0)
           : a == 1 ? ((i == 3 || i == 5 || i == 8) ? 1 : (i == 4 || i == 6 || i == 7) ? -1 : 0)
                    : 0;
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
};

template <>
struct Lat<19> {
  static constexpr int D = 3, NS = 6;
  __host__ __device__ static constexpr int c(int i, int a) {
    return a == 0   ? ((i == 1 || i == 7 || i == 9 || i == 11 || i == 13)    ? 1
                       : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1
                                                                               : 0)
           : a == 1 ? ((i == 3 || i == 7 || i == 10 || i == 15 || i == 17)   ? 1
                       : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18)  ? -1
                                                                               : 0)
                    : ((i == 5 || i == 11 || i == 14 || i == 15 || i == 18)  ? 1
                       : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1
                                                                                : 0);
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
  }
};

template <>
struct Lat<27> {
  static constexpr int D = 3, NS = 6;
  // base-3 code (cx+1) + 3 (cy+1) + 9 (cz+1) of each velocity, in lbm.h order
  __host__ __device__ static constexpr int code(int i) {
    return i == 0 ? 13 : i == 1 ? 14 : i == 2 ? 12 : i == 3 ? 16 : i == 4 ? 10 : i == 5 ? 22 : i == 6 ? 4 : i == 7 ? 17 : i == 8 ? 9 : i == 9 ? 11 : i == 10 ? 15 : i == 11 ? 23 : i == 12 ? 3 : i == 13 ? 5 : i == 14 ? 21 : i == 15 ? 25 : i == 16 ? 1 : i == 17 ? 7 : i == 18 ? 19 : i == 19 ? 26 : i == 20 ? 0 : i == 21 ? 8 : i == 22 ? 18 : i == 23 ? 20 : i == 24 ? 6 : i == 25 ? 24 : 2;
  }
  __host__ __device__ static constexpr int c(int i, int a) {
    return (a == 0 ? code(i) % 3 : (a == 1 ? code(i) / 3 % 3 : code(i) / 9)) - 1;
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 8.0 / 27.0 : (i <= 6 ? 2.0 / 27.0 : (i <= 18 ? 1.0 / 54.0 : 1.0 / 216.0));
  }
};

__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }

// Run-time lookup of c_{i,a} and w_i for a velocity index known only at run
// time (a lane's share of the directions): c_{i,a} + 1 packed in two bits per
// velocity; the weights depend on |c_i|^2, i.e. on the index range (every
// lattice lists its velocities by increasing length).
template <int Q>
struct LatRt {
  __host__ __device__ static constexpr uint64_t pack(int a) {
    uint64_t m = 0;
    for (int i = 0; i < Q; ++i) m |= (uint64_t)(Lat<Q>::c(i, a) + 1) << (2 * i);
    return m;
  }
  __device__ static __forceinline__ int c(int i, int a) {
    constexpr uint64_t X = pack(0), Y = pack(1), Z = pack(2);
    const uint64_t m = a == 0 ? X : (a == 1 ? Y : Z);
    return (int)((m >> (2 * i)) & 3u) - 1;
  }
  template <class R>
  __device__ static __forceinline__ R w(int i) {
    constexpr int D = Lat<Q>::D;
    return i == 0 ? R(Lat<Q>::w(0))
                  : (i <= 2 * D ? R(Lat<Q>::w(1)) : ((Q == 27 && i > 18) ? R(Lat<Q>::w(19)) : R(Lat<Q>::w(2 * D + 1))));
  }
};

// index of S_ab in the packed strain-rate vector (xx,yy,xy | xx,yy,zz,xy,yz,xz)
template <int D>
__host__ __device__ constexpr int sidx(int a, int b) {
  return a == b ? a
                : (D == 2 ? 2
                          : ((a + b == 1) ? 3 : ((a + b == 3) ? 4 : 5)));
}

// ----------------------------------------------------------------- storage
template <class S>
struct Sto;
template <>
struct Sto<double> {
  using R = double;
  __device__ static __forceinline__ R ld(const double* p) { return *p; }
  __device__ static __forceinline__ double cv(R v) { return v; }
};
template <>
struct Sto<float> {
  using R = float;
  __device__ static __forceinline__ R ld(const float* p) { return *p; }
  __device__ static __forceinline__ float cv(R v) { return v; }
};
template <>
struct Sto<__nv_bfloat16> {
  using R = float;
  __device__ static __forceinline__ R ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  __device__ static __forceinline__ __nv_bfloat16 cv(R v) { return __float2bfloat16_rn(v); }
};

// Programmatic dependent launch of the step's kernels (launched so where
// *Args::chain is set): once every block of a kernel has its inputs, the
// successor's blocks may start, and load what no kernel of the step writes
// (tables, neighbour lists) before they wait for its end here.  Before the
// wait a kernel neither reads the state nor writes anything, and no kernel
// lets the next one start before it: at most two of a chain are resident.
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Index of the launch segment that holds block b, given the segments' first
// blocks in order (uniform over the block).
__device__ __forceinline__ int segment_of(const uint32_t* first, int n, unsigned b) {
  int s = 0;
  for (int k = 1; k < n; ++k)
    if (b >= first[k]) s = k;
  return s;
}

// The compute type's one of two launch constants.
template <class R>
__device__ __forceinline__ auto& pick(const double& d, const float& f) {
  if constexpr (sizeof(R) == 8) return d;
  else return f;
}
template <class R>
__device__ __forceinline__ auto& pick(const Relax& d, const Relax32& f) {
  if constexpr (sizeof(R) == 8) return d;
  else return f;
}
template <class R>
__device__ __forceinline__ auto& pick(const GhostUnits<double>& d, const GhostUnits<float>& f) {
  if constexpr (sizeof(R) == 8) return d;
  else return f;
}
template <class R>
using RelaxOf = std::conditional_t<sizeof(R) == 8, Relax, Relax32>;

// ----------------------------------------------------------------- physics
// g^eq_i for density deviation rp = rho - rho_off
template <int Q, class R>
__device__ __forceinline__ R geq(int i, R rp, R rho, const R* u, R usq) {
  using LT = Lat<Q>;
  R cu = R(0);
#pragma unroll
  for (int a = 0; a < LT::D; ++a) cu += R(LT::c(i, a)) * u[a];
  return R(LT::w(i)) * (rp + rho * (R(3) * cu + R(4.5) * cu * cu - R(1.5) * usq));
}

// Guo forcing term (1 - omega/2) w_i [3 (c_i - u) + 9 (c_i.u) c_i] . F
template <int Q, class R>
__device__ __forceinline__ R guo(int i, R omega, const R* u, const R* F) {
  using LT = Lat<Q>;
  R cu = R(0), cF = R(0), uF = R(0);
#pragma unroll
  for (int a = 0; a < LT::D; ++a) {
    cu += R(LT::c(i, a)) * u[a];
    cF += R(LT::c(i, a)) * F[a];
    uF += u[a] * F[a];
  }
  return (R(1) - R(0.5) * omega) * R(LT::w(i)) * (R(3) * (cF - uF) + R(9) * cu * cF);
}

// rho deviation and first moment of a pdf set
template <int Q, class R>
__device__ __forceinline__ void raw_moments(const R* g, R& rp, R* j) {
  using LT = Lat<Q>;
  rp = R(0);
  j[0] = j[1] = j[2] = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    rp += g[i];
#pragma unroll
    for (int a = 0; a < LT::D; ++a) {
      if (LT::c(i, a) > 0) j[a] += g[i];
      if (LT::c(i, a) < 0) j[a] -= g[i];
    }
  }
}

// Pre-collision moments from a stored post-collision set: u = (j - F/2)/rho,
// f^neq = (g - g^eq - F_i) r1w, r1w = 1 / (1 - omega), S_ab = -(3 omega / 2 rho) sum c_a c_b f^neq.
// g^eq per pair of opposite velocities (c.u changes sign: the even part is
// shared); without FORCE the forcing terms are left out at compile time.
template <int Q, class R, bool WANT_S, bool FORCE = true>
__device__ __forceinline__ void post_moments(const R* g, R omega, R r1w, R rho_off, const R* F, R& rp, R* u,
                                             R* fneq, R* S) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  R j[3];
  raw_moments<Q, R>(g, rp, j);
  const R rho = rho_off + rp;
  const R inv = R(1) / rho;
  u[0] = u[1] = u[2] = R(0);
#pragma unroll
  for (int a = 0; a < D; ++a) u[a] = (FORCE ? j[a] - R(0.5) * F[a] : j[a]) * inv;
  R usq = R(0);
#pragma unroll
  for (int a = 0; a < D; ++a) usq += u[a] * u[a];
  const R base = rp - R(1.5) * rho * usq;
  {
    R f0 = g[0] - R(LT::w(0)) * base;
    if (FORCE) f0 -= guo<Q, R>(0, omega, u, F);
    fneq[0] = f0 * r1w;
  }
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    R cu = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (LT::c(i, a) > 0) cu += u[a];
      if (LT::c(i, a) < 0) cu -= u[a];
    }
    const R w = R(LT::w(i));
    const R even = w * (base + R(4.5) * rho * cu * cu);
    const R odd = w * R(3) * rho * cu;
    R fa = g[i] - (even + odd), fb = g[i + 1] - (even - odd);
    if (FORCE) {
      fa -= guo<Q, R>(i, omega, u, F);
      fb -= guo<Q, R>(i + 1, omega, u, F);
    }
    fneq[i] = fa * r1w;
    fneq[i + 1] = fb * r1w;
  }
  if (WANT_S) {
    const R pre = -R(1.5) * omega * inv;
#pragma unroll
    for (int s = 0; s < LT::NS; ++s) S[s] = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
#pragma unroll
      for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = a; b < D; ++b) {
          const int cc = LT::c(i, a) * LT::c(i, b);
          if (cc > 0) S[sidx<D>(a, b)] += fneq[i];
          if (cc < 0) S[sidx<D>(a, b)] -= fneq[i];
        }
    }
#pragma unroll
    for (int s = 0; s < LT::NS; ++s) S[s] *= pre;
  }
}

// ----------------------------------------------------------------- FP64 arithmetic
// GB300 issues an FP64 instruction of a warp over about 19 cycles of its SM,
// so the FP64 kernels are bound by the number of FP64 instructions, and these
// forms of the moments, the collision and post_moments are written for fewest
// of them: c.j instead of c.u (one reciprocal, no velocity), every uniform
// factor a constant operand (Relax), each pair of opposite velocities as two
// fused multiply-adds on its two values, signs flipped on the integer pipe.
// With one-warp blocks (kScBlock), per coarse step of two-level flows: forced
// D3Q19, 1.5e5 elements, 293 -> 211 us; D2Q9, 1,800 elements, 67 -> 47 us.
template <int Q>
__host__ __device__ constexpr int wclass(int i) {
  return Lat<Q>::c(i, 0) * Lat<Q>::c(i, 0) + Lat<Q>::c(i, 1) * Lat<Q>::c(i, 1) + Lat<Q>::c(i, 2) * Lat<Q>::c(i, 2);
}

// x with its sign flipped when `neg`
__device__ __forceinline__ double flip(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000 : 0), __double2loint(x));
}

// sum of the pdfs and first moment: the x moment shares its two half sums
// with the total, the other axes take the differences of opposite pdfs
template <int Q>
__device__ __forceinline__ void raw_moments64(const double* g, double& rp, double* j) {
  using LT = Lat<Q>;
  double sp = 0, sm = 0, s0 = g[0], s1 = 0;  // short chains: a lone warp waits for each sum
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (LT::c(i, 0) > 0) sp += g[i];
    else if (LT::c(i, 0) < 0) sm += g[i];
    else if (i & 1) s0 += g[i];
    else s1 += g[i];
  }
  rp = (sp + sm) + (s0 + s1);
  j[0] = sp - sm;
  j[1] = j[2] = 0;
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    if (LT::c(i, 1) == 0 && LT::c(i, 2) == 0) continue;
    const double m = g[i] - g[i + 1];
#pragma unroll
    for (int a = 1; a < LT::D; ++a) {
      if (LT::c(i, a) > 0) j[a] += m;
      if (LT::c(i, a) < 0) j[a] -= m;
    }
  }
}

// c_i . v
template <int Q>
__device__ __forceinline__ double cdot(int i, const double* v) {
  using LT = Lat<Q>;
  double s = 0;
#pragma unroll
  for (int a = 0; a < LT::D; ++a) {
    if (LT::c(i, a) > 0) s += v[a];
    if (LT::c(i, a) < 0) s -= v[a];
  }
  return s;
}

// BGK collision of one element in place (bgk_collide): with J = rho u,
//   g_i := (1 - omega) g_i + omega w [rp - 3/2 J.J / rho + 9/2 (c.J)^2 / rho + 3 c.J] + Guo
template <int Q, bool FORCE>
__device__ __forceinline__ void bgk_collide64(double (&g)[Q], const Relax& rx, double rho_off, const double* F) {
  using LT = Lat<Q>;
  constexpr int D = LT::D, NC = Q == 27 ? 4 : 3;
  double rp, J[3];
  raw_moments64<Q>(g, rp, J);
  if (FORCE) {
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = fma(0.5, F[a], J[a]);
  }
  const double inv = 1.0 / (rho_off + rp);
  double jj = 0, jF = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    jj = fma(J[a], J[a], jj);
    if (FORCE) jF = fma(J[a], F[a], jF);
  }
  const double base = fma(-1.5 * inv, jj, rp);
  const double uF = FORCE ? jF * inv : 0.0;
  double b[NC], kq[NC], kf[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    b[c] = FORCE ? fma(rx.eq(c), base, -rx.force[c] * uF) : rx.eq(c) * base;
    kq[c] = c ? rx.quad(c) * inv : 0.0;
    kf[c] = FORCE && c ? 3.0 * rx.force[c] * inv : 0.0;
  }
  g[0] = fma(rx.keep, g[0], b[0]);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const int c = wclass<Q>(i);
    const double cJ = cdot<Q>(i, J);
    if (FORCE) {
      const double cF = cdot<Q>(i, F);
      const double ev = fma(cJ, fma(kq[c], cJ, kf[c] * cF), b[c]);
      const double od = fma(rx.lin(c), cJ, rx.force[c] * cF);
      g[i] = fma(rx.keep, g[i], ev + od);
      g[i + 1] = fma(rx.keep, g[i + 1], ev - od);
    } else {
      const double ev = fma(kq[c] * cJ, cJ, b[c]);
      g[i] = fma(rx.keep, g[i], fma(rx.lin(c), cJ, ev));
      g[i + 1] = fma(rx.keep, g[i + 1], fma(-rx.lin(c), cJ, ev));
    }
  }
}

// post_moments with the strain rate
template <int Q, bool FORCE>
__device__ __forceinline__ void post_moments64(const double* g, const Relax& rx, double rho_off, const double* F,
                                               double& rp, double* u, double* fneq, double* S) {
  using LT = Lat<Q>;
  constexpr int D = LT::D, NS = LT::NS, NC = Q == 27 ? 4 : 3;
  double J[3];
  raw_moments64<Q>(g, rp, J);
  if (FORCE) {
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = fma(-0.5, F[a], J[a]);
  }
  const double inv = 1.0 / (rho_off + rp);
  double jj = 0, uF = 0;
  u[0] = u[1] = u[2] = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    u[a] = J[a] * inv;
    jj = fma(J[a], u[a], jj);
    if (FORCE) uF = fma(u[a], F[a], uF);
  }
  const double base = fma(-1.5, jj, rp);
  double b[NC], kq[NC], kf[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    b[c] = FORCE ? fma(rx.nforce[c], uF, -rx.neq(c) * base) : -rx.neq(c) * base;
    kq[c] = c ? -rx.nquad(c) * inv : 0.0;
    kf[c] = FORCE && c ? -3.0 * rx.nforce[c] * inv : 0.0;
  }
  fneq[0] = fma(rx.r1w, g[0], b[0]);
#pragma unroll
  for (int s = 0; s < NS; ++s) S[s] = 0;
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const int c = wclass<Q>(i);
    const double cJ = cdot<Q>(i, J);
    if (FORCE) {
      const double cF = cdot<Q>(i, F);
      const double ev = fma(cJ, fma(kq[c], cJ, kf[c] * cF), b[c]);
      const double od = fma(rx.nlin(c), cJ, rx.nforce[c] * cF);
      fneq[i] = fma(rx.r1w, g[i], ev - od);
      fneq[i + 1] = fma(rx.r1w, g[i + 1], ev + od);
    } else {
      const double ev = fma(kq[c] * cJ, cJ, b[c]);
      fneq[i] = fma(rx.r1w, g[i], fma(-rx.nlin(c), cJ, ev));
      fneq[i + 1] = fma(rx.r1w, g[i + 1], fma(rx.nlin(c), cJ, ev));
    }
    const double ps = fneq[i] + fneq[i + 1];
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int e = a; e < D; ++e) {
        const int cc = LT::c(i, a) * LT::c(i, e);
        if (cc > 0) S[sidx<D>(a, e)] += ps;
        if (cc < 0) S[sidx<D>(a, e)] -= ps;
      }
  }
  const double pre = rx.strain * inv;
#pragma unroll
  for (int s = 0; s < NS; ++s) S[s] *= pre;
}

// ----------------------------------------------------------------- GFC source records
// Record of one source (compute type, mom_stride(Q) values, 16-byte aligned
// groups): f^neq[Q] padded to a multiple of 4, then rho - rho_off, u[D], S[nS],
// padding.  Vector loads/stores move a record in 8 (float) or 16 (double) pieces.
template <int Q>
struct RecLayout {
  static constexpr int D = Lat<Q>::D, NS = Lat<Q>::NS;
  static constexpr int FN = 0;
  static constexpr int RP = (Q + 3) / 4 * 4;
  static constexpr int U = RP + 1;
  static constexpr int SS = U + D;
  static constexpr int END = SS + NS;
  static constexpr int STRIDE = mom_stride(Q);
  static_assert(END <= STRIDE && STRIDE % 4 == 0, "moment record too long");
};

__device__ __forceinline__ void ld4(const float* p, float* o) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  o[0] = v.x;
  o[1] = v.y;
  o[2] = v.z;
  o[3] = v.w;
}
__device__ __forceinline__ void ld4(const double* p, double* o) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  o[0] = a.x;
  o[1] = a.y;
  o[2] = b.x;
  o[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(double* p, const double* v) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

// Interpolation step 1 (Sec. 2.2) for one source: its record from its stored
// (post-collision) pdfs g.
template <int Q, class R, bool FORCE>
__device__ __forceinline__ void source_record(const R (&g)[Q], const RelaxOf<R>& rx, R rho_off, const R* F,
                                              R (&rec)[RecLayout<Q>::STRIDE]) {
  using RL = RecLayout<Q>;
  constexpr int D = Lat<Q>::D, NS = Lat<Q>::NS;
#pragma unroll
  for (int f = 0; f < RL::STRIDE; ++f) rec[f] = R(0);
  R rp, u[3], fneq[Q], Sv[NS];
  if constexpr (sizeof(R) == 8) post_moments64<Q, FORCE>(g, rx, rho_off, F, rp, u, fneq, Sv);
  else post_moments<Q, R, true, FORCE>(g, rx.omega, rx.r1w, rho_off, F, rp, u, fneq, Sv);
#pragma unroll
  for (int q = 0; q < Q; ++q) rec[RL::FN + q] = fneq[q];
  rec[RL::RP] = rp;
#pragma unroll
  for (int b = 0; b < D; ++b) rec[RL::U + b] = u[b];
#pragma unroll
  for (int s = 0; s < NS; ++s) rec[RL::SS + s] = Sv[s];
}

// rec := (prev + rec) / 2; the whole previous record is read before the
// caller's first store (the compiler cannot tell the records apart and would
// otherwise serialise loads and stores)
template <int Q, class R>
__device__ __forceinline__ void mean_record(const R* __restrict__ prev, R (&rec)[RecLayout<Q>::STRIDE]) {
  using RL = RecLayout<Q>;
  R pv[RL::STRIDE];
#pragma unroll
  for (int f = 0; f < RL::END; f += 4) ld4(prev + f, pv + f);
#pragma unroll
  for (int f = 0; f < RL::END; ++f) rec[f] = R(0.5) * (pv[f] + rec[f]);
}

template <int Q, class R>
__device__ __forceinline__ void store_record(R* __restrict__ out, const R (&rec)[RecLayout<Q>::STRIDE]) {
#pragma unroll
  for (int f = 0; f < RecLayout<Q>::END; f += 4) st4(out + f, rec + f);
}

// Record index of element e among its level's GhostFromCoarser sources, -1 if
// it is none.  Mask words are per 32 slots: one broadcast load for a warp of
// consecutive elements.
__device__ __forceinline__ int64_t source_index(const SourceTable& so, int64_t e) {
  const uint32_t m = __ldg(so.mask + (e >> 5));
  const uint32_t bit = (uint32_t)e & 31u;
  if (!((m >> bit) & 1u)) return -1;
  return (int64_t)__ldg(so.first + (e >> 5)) + __popc(m & ((1u << bit) - 1u));
}

// Stream-collide epilogue for a GhostFromCoarser source among the processed
// elements: g are the element's new values before rounding to storage; the
// record is taken from the values as stored, so it equals what
// k_source_moments computes from the stored state.
template <int Q, class S, bool FORCE>
__device__ __forceinline__ void source_out(const SourceTable& so, void* rec_out, int64_t e,
                                           const typename Sto<S>::R (&g)[Q], const RelaxOf<typename Sto<S>::R>& rx,
                                           typename Sto<S>::R rho_off, const typename Sto<S>::R* F) {
  using R = typename Sto<S>::R;
  using RL = RecLayout<Q>;
  const int64_t k = source_index(so, e);
  if (k < 0) return;
  R gs[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const S v = Sto<S>::cv(g[q]);
    gs[q] = Sto<S>::ld(&v);
  }
  R rec[RL::STRIDE];
  source_record<Q, R, FORCE>(gs, rx, rho_off, F, rec);
  store_record<Q, R>(static_cast<R*>(rec_out) + k * RL::STRIDE, rec);
}

// ----------------------------------------------------------------- stream + collide
// LBM_SC_STREAM: streaming (evict-first) hints on the use-once neighbour
// indices and on the stores.
#ifndef LBM_SC_STREAM
#define LBM_SC_STREAM 1
#endif

__device__ __forceinline__ uint32_t ld_once(const uint32_t* p) {
#if LBM_SC_STREAM
  return __ldcs(p);
#else
  return __ldg(p);
#endif
}
__device__ __forceinline__ void st_once(double* p, double v) {
#if LBM_SC_STREAM
  __stcs(p, v);
#else
  *p = v;
#endif
}
__device__ __forceinline__ void st_once(float* p, float v) {
#if LBM_SC_STREAM
  __stcs(p, v);
#else
  *p = v;
#endif
}
__device__ __forceinline__ void st_once(__nv_bfloat16* p, __nv_bfloat16 v) {
#if LBM_SC_STREAM
  __stcs(reinterpret_cast<unsigned short*>(p), __bfloat16_as_ushort(v));
#else
  *p = v;
#endif
}

// BGK collision (Eq. bgk) of one element in place, with Guo forcing, using the
// symmetry of each velocity pair (i, opp(i)): c.u and c.F change sign, so the
// even part of f^eq (and of the forcing term) is shared and the odd part flips.
template <int Q, class R, bool FORCE>
__device__ __forceinline__ void bgk_collide(R (&g)[Q], const RelaxOf<R>& rx, R rho_off, const R* F) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  if constexpr (sizeof(R) == 8) {
    bgk_collide64<Q, FORCE>(g, rx, rho_off, F);
    return;
  }
  const R om = rx.omega;
  R rp, j[3];
  raw_moments<Q, R>(g, rp, j);
  const R rho = rho_off + rp;
  const R inv = R(1) / rho;
  R u[3] = {R(0), R(0), R(0)};
#pragma unroll
  for (int b = 0; b < D; ++b) u[b] = (j[b] + (FORCE ? R(0.5) * F[b] : R(0))) * inv;
  R usq = R(0), uF = R(0);
#pragma unroll
  for (int b = 0; b < D; ++b) {
    usq += u[b] * u[b];
    if (FORCE) uF += u[b] * F[b];
  }
  const R base = rp - R(1.5) * rho * usq;  // even part without the (c.u)^2 term, per unit weight
  const R fpre = FORCE ? (R(1) - R(0.5) * om) : R(0);
  {
    R geq0 = R(LT::w(0)) * base;
    R gi = g[0] + om * (geq0 - g[0]);
    if (FORCE) gi += fpre * R(LT::w(0)) * (-R(3) * uF);
    g[0] = gi;
  }
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    R cu = R(0), cF = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      if (LT::c(i, b) > 0) {
        cu += u[b];
        if (FORCE) cF += F[b];
      }
      if (LT::c(i, b) < 0) {
        cu -= u[b];
        if (FORCE) cF -= F[b];
      }
    }
    const R w = R(LT::w(i));
    const R even = w * (base + R(4.5) * rho * cu * cu);
    const R odd = w * R(3) * rho * cu;
    R a = g[i] + om * (even + odd - g[i]);
    R b = g[i + 1] + om * (even - odd - g[i + 1]);
    if (FORCE) {
      const R fe = fpre * w * (R(9) * cu * cF - R(3) * uF);
      const R fo = fpre * w * R(3) * cF;
      a += fe + fo;
      b += fe - fo;
    }
    g[i] = a;
    g[i + 1] = b;
  }
}

// FP64 storage: one warp per block.  A warp holds its SM's FP64 pipe for about
// 120 x 19 cycles, so a launch takes as long as the SM with the most warps,
// and small blocks spread a small level over all SMs (D2Q9, 1,800 elements:
// 7 blocks of 256 on 7 SMs before).  12 to 24 warps per SM keep the pipe busy,
// and bounds of 24, 16 and 12 blocks (D2Q9, D3Q19, D3Q27) leave every kernel
// the registers it takes, 64, 114 and 148 at most; 80 for D3Q19 spilled.
template <class S>
constexpr int kScBlock = sizeof(S) == 8 ? 32 : 256;
template <int Q>
constexpr int kScMinb64 = Q == 27 ? 12 : Q == 19 ? 16 : 24;

// Collision, store and source record of one element from its pulled pdfs.
template <int Q, class S, bool FORCE, bool MOMS>
__device__ __forceinline__ void sc_finish(const ScArgs& a, const ScSeg& sg, int64_t e,
                                          typename Sto<S>::R (&g)[Q]) {
  using R = typename Sto<S>::R;
  constexpr int D = Lat<Q>::D;
  const size_t N = (size_t)a.Ntot;
  R F[3] = {R(0), R(0), R(0)};
  if (FORCE) {
    const R* __restrict__ fp = static_cast<const R*>(a.force) + e;
#pragma unroll
    for (int c = 0; c < D; ++c) F[c] = fp[c * N];
  }
  const R rho_off = pick<R>(a.rho_off, a.rho_off32);
  const auto& rx = pick<R>(a.rx[sg.level], sg.rx);
  let_next_start();
  bgk_collide<Q, R, FORCE>(g, rx, rho_off, F);
  S* __restrict__ dst = static_cast<S*>(sg.dst) + e;
#pragma unroll
  for (int i = 0; i < Q; ++i) st_once(dst + i * N, Sto<S>::cv(g[i]));
  if (MOMS)
    if (sg.rec_out) source_out<Q, S, FORCE>(a.sources, sg.rec_out, e, g, rx, rho_off, F);
}

// the incoming value of a link with a boundary code: the inlet's term on top
// of the bounce-back value, or the precomputed boundary value
template <class R>
__device__ __forceinline__ R link_value(const ScArgs& a, const ScSeg& sg, int i, uint32_t n, R back) {
  if (n & NB_BOUNCE) return back + R(a.inlet[i] * (double)sg.uin) * (a.inlet_s ? R(a.inlet_s[n & NB_INDEX]) : R(1));
  return static_cast<const R*>(a.side)[n & NB_INDEX];
}

// Pull streaming f_i(x) = f*_i(x - c_i) (Sec. 2.1, Eq. lbe) of interior bricks:
// the pull source of link i is located by the brick's neighbour row instead
// of the per-element neighbour list.  Each group of 64 threads takes one brick,
// thread l its element at z-curve position l; blocks are issued in brick
// order, so the bricks in flight stay a compact window of the level and their
// neighbours' lines are still in L2 when gathered.  The thread's Q-1
// link-table entries (slot, position) are loaded into registers, lanes 0..26
// of each warp load the brick's 27-entry neighbour row in one coalesced
// access, and every link takes its row entry by a warp shuffle, so all pdf
// gathers issue after two loads.  The element's HBM traffic is its Q pdf reads
// and Q writes.
// the link-table entries of position l, and lane's entry of the brick's row
template <int Q>
struct BrickLinks {
  uint32_t tw[Q / 2];  // (Q-1)/2 words of two 16-bit entries
  int32_t row;
  __device__ __forceinline__ void load(const uint16_t* tab, const int32_t* nb, int64_t b, int l, int lane) {
#pragma unroll
    for (int k = 0; k < Q / 2; ++k)
      tw[k] = (uint32_t)__ldg(tab + (2 * k) * 64 + l) | ((uint32_t)__ldg(tab + (2 * k + 1) * 64 + l) << 16);
    row = lane < 27 ? __ldg(nb + b * 27 + lane) : 0;
  }
  __device__ __forceinline__ uint32_t entry(int i) const { return (tw[(i - 1) >> 1] >> (((i - 1) & 1) * 16)) & 0xffffu; }
};

template <int Q, class S>
__device__ __forceinline__ void pull_interior(const ScArgs& a, const ScSeg& sg, const BrickLinks<Q>& k, int64_t first,
                                              int l, typename Sto<S>::R (&g)[Q]) {
  const size_t N = (size_t)a.Ntot;
  const S* __restrict__ src = static_cast<const S*>(sg.src) + first;
  g[0] = Sto<S>::ld(src + l);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const uint32_t v = k.entry(i);
    const int32_t r = __shfl_sync(0xffffffffu, k.row, (int)(v >> 6));
    g[i] = Sto<S>::ld(src + (int64_t)(i * N) + r + (v & 63));
  }
}

// Pull of the elements that read ghosts or boundary values: boundary bricks (a
// complete brick whose neighbour brick behind some link is not complete: row
// entry kBrickMissing) and the elements of the neighbour-list range, all of
// whose links go through the list.  Every link is first resolved to one
// 32-bit offset from src + i N + first: the brick-table entry, or the
// element's neighbour-list code turned into a pull (n - first), its own
// opposite slot (bounce-back, and the inlet's base value: (opp(i) - i) N + l),
// or, for a boundary value, that same valid slot, the value being substituted
// afterwards.  So all codes are loaded before any is used, and the gathers
// need no branch.  |offsets| < 2^30 + 64 since Ntot < 2^30.
template <int Q, class S>
__device__ __forceinline__ void pull_rest(const ScArgs& a, const ScSeg& sg, int32_t (&off)[Q], uint32_t miss,
                                          int64_t first, int l, typename Sto<S>::R (&g)[Q]) {
  const size_t N = (size_t)a.Ntot;
  const S* __restrict__ src = static_cast<const S*>(sg.src) + first;
  uint32_t patch = 0;  // links whose value gets an inlet term or a substitute
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
  g[0] = Sto<S>::ld(src + l);
#pragma unroll
  for (int i = 1; i < Q; ++i) g[i] = Sto<S>::ld(src + (int64_t)(i * N) + off[i]);
  // the inlet term or the precomputed boundary value, from the link's code
  // read again
  if (patch) {
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if (!((patch >> i) & 1u)) continue;
      g[i] = link_value(a, sg, i, __ldg(a.nbr + (size_t)(i - 1) * N + first + l), g[i]);
    }
  }
}

// Minimum blocks of 256 per SM (FP32, BF16).  D3Q19 and D2Q9: five, 48
// registers (boundary bricks alone 4.66 against 4.38 TB/s at four); D3Q27:
// four for interior bricks, three for the rest.
template <int Q, class S>
constexpr int kIntMinb = sizeof(S) == 8 ? kScMinb64<Q> : Q <= 19 ? 5 : 4;
template <int Q, class S>
constexpr int kRestMinb = sizeof(S) == 8 ? kScMinb64<Q> : Q <= 19 ? 5 : 3;

template <int Q, class S, bool FORCE, bool MOMS>
__global__ void __launch_bounds__(kScBlock<S>, kIntMinb<Q, S>) k_sc_interior(const __grid_constant__ ScArgs a) {
  const int seg = segment_of(a.first, a.nseg, blockIdx.x);
  const ScSeg& sg = a.seg[seg];
  const int64_t t = (int64_t)(blockIdx.x - a.first[seg]) * kScBlock<S> + threadIdx.x;
  const int l = (int)t & 63, lane = threadIdx.x & 31;
  // the brick index is uniform over each warp (64 threads per brick), so the
  // exit below and the shuffles run with whole warps
  const int64_t b = t >> 6;
  if (b >= sg.n) return;
  BrickLinks<Q> k;
  k.load(a.tab, sg.nb, b, l, lane);
  const int64_t first = sg.begin + b * 64;
  typename Sto<S>::R g[Q];
  wait_for_previous();
  pull_interior<Q, S>(a, sg, k, first, l, g);
  sc_finish<Q, S, FORCE, MOMS>(a, sg, first + l, g);
}

// Everything that reads ghosts or boundary values: boundary bricks and (LIST)
// the elements of the neighbour-list range (incomplete bricks, the processed
// ghost layers), in one launch.
template <int Q, class S, bool FORCE, bool MOMS, bool LIST>
__global__ void __launch_bounds__(kScBlock<S>, kRestMinb<Q, S>) k_sc_rest(const __grid_constant__ ScArgs a) {
  const int seg = segment_of(a.first, a.nseg, blockIdx.x);
  const ScSeg& sg = a.seg[seg];
  const int64_t t = (int64_t)(blockIdx.x - a.first[seg]) * kScBlock<S> + threadIdx.x;
  const size_t N = (size_t)a.Ntot;
  int32_t off[Q];
  uint32_t miss = 0;
  int64_t first;
  int l = 0;
  if (LIST && sg.list) {
    if (t >= sg.n) return;
    const int64_t lin = sg.begin + t;
    first = lin + (lin >= sg.hole_at ? sg.hole_len : 0);
#pragma unroll
    for (int i = 1; i < Q; ++i) off[i] = (int32_t)ld_once(a.nbr + (size_t)(i - 1) * N + first);
    miss = ~0u;
  } else {
    // the brick index is uniform over each warp: whole warps exit or shuffle
    const int64_t b = t >> 6;
    if (b >= sg.n) return;
    l = (int)t & 63;
    BrickLinks<Q> k;
    k.load(a.tab, sg.nb, b, l, threadIdx.x & 31);
    first = sg.begin + b * 64;
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
  typename Sto<S>::R g[Q];
  wait_for_previous();
  pull_rest<Q, S>(a, sg, off, miss, first, l, g);
  sc_finish<Q, S, FORCE, MOMS>(a, sg, first + l, g);
}

// BF16 interior bricks, two neighbouring elements per thread: lane m of the
// brick's warp takes z-curve positions 2m and 2m+1, which differ only in the
// lowest x bit, so they sit next to each other in every direction array.  A
// link with c_x = 0 pulls both sources from one brick slot at positions l'
// and l'+1 (the mesh builder checks this on the link table), one 32-bit
// bfloat16 pair load at an even element index; links with c_x != 0 take two
// single loads.  The 19 results are written as bfloat16 pairs, rounded by one
// packed conversion each.  Same pull and BGK collision as the one-element
// kernel, element by element.
// 128-thread blocks (four bricks), 1024 threads per SM (64 registers) for
// D2Q9 / D3Q19, 768 for D3Q27 (which spills at 1024).  Measured on the
// sphere's finest level: 5.46 TB/s against 5.37 with 256-thread blocks and
// 4.91 with 512; 1280 threads per SM (48 registers) spilled and was slower.
// plain stores (no evict-first hint) measured 0.3% faster for this kernel
#ifndef LBM_PAIR_STCS
#define LBM_PAIR_STCS 0
#endif
#ifndef LBM_BR_PAIR_BLOCK
#define LBM_BR_PAIR_BLOCK 128
#endif
#ifndef LBM_BR_PAIR_MINB_Q19
#define LBM_BR_PAIR_MINB_Q19 (1024 / LBM_BR_PAIR_BLOCK)
#endif
#define LBM_BR_PAIR_MINB(Q) ((Q) > 19 ? 768 / LBM_BR_PAIR_BLOCK : LBM_BR_PAIR_MINB_Q19)
template <int Q, bool FORCE>
__global__ void __launch_bounds__(LBM_BR_PAIR_BLOCK, LBM_BR_PAIR_MINB(Q)) k_sc_interior_pair(const __grid_constant__ ScArgs a) {
  using S = __nv_bfloat16;
  using R = float;
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  constexpr int BPB = LBM_BR_PAIR_BLOCK / 32;
  const int m = threadIdx.x & 31;
  const ScSeg& sg = a.seg[0];  // issue bound: one segment per launch, no search
  // one brick per warp: the exit below and the shuffles run with whole warps
  const int64_t b = (int64_t)blockIdx.x * BPB + (threadIdx.x >> 5);
  if (b >= sg.n) return;
  const int32_t row = m < 27 ? __ldg(sg.nb + b * 27 + m) : 0;
  const size_t N = (size_t)a.Ntot;
  const int64_t first = sg.begin + b * 64;
  const S* __restrict__ src = static_cast<const S*>(sg.src) + first;
  S* __restrict__ dst = static_cast<S*>(sg.dst) + first + 2 * m;
  // the link-table entries of positions 2m (low half) and 2m+1 (high half)
  const uint32_t* __restrict__ tab2 = reinterpret_cast<const uint32_t*>(a.tab);
  R g0[Q], g1[Q];
  {
    const __nv_bfloat162 p = *reinterpret_cast<const __nv_bfloat162*>(src + 2 * m);
    g0[0] = __low2float(p);
    g1[0] = __high2float(p);
  }
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const uint32_t tw = __ldg(tab2 + (i - 1) * 32 + m);
    const S* base = src + (int64_t)(i * N);
    if (LT::c(i, 0) == 0) {
      const uint32_t v = tw & 0xffffu;
      const int32_t r = __shfl_sync(0xffffffffu, row, (int)(v >> 6));
      const __nv_bfloat162 p = *reinterpret_cast<const __nv_bfloat162*>(base + (r + (int32_t)(v & 63)));
      g0[i] = __low2float(p);
      g1[i] = __high2float(p);
    } else {
      const uint32_t v0 = tw & 0xffffu, v1 = tw >> 16;
      const int32_t r0 = __shfl_sync(0xffffffffu, row, (int)(v0 >> 6));
      const int32_t r1 = __shfl_sync(0xffffffffu, row, (int)(v1 >> 6));
      // signed sums: a neighbour brick stored before this one has r < 0
      g0[i] = __bfloat162float(base[r0 + (int32_t)(v0 & 63)]);
      g1[i] = __bfloat162float(base[r1 + (int32_t)(v1 & 63)]);
    }
  }
  R F0[3] = {R(0), R(0), R(0)}, F1[3] = {R(0), R(0), R(0)};
  if (FORCE) {
    const R* __restrict__ fp = static_cast<const R*>(a.force) + first + 2 * m;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const float2 f = *reinterpret_cast<const float2*>(fp + c * N);
      F0[c] = f.x;
      F1[c] = f.y;
    }
  }
  bgk_collide<Q, R, FORCE>(g0, sg.rx, a.rho_off32, F0);
  bgk_collide<Q, R, FORCE>(g1, sg.rx, a.rho_off32, F1);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(g0[i], g1[i]);
#if LBM_SC_STREAM && LBM_PAIR_STCS
    __stcs(reinterpret_cast<unsigned int*>(dst + i * N), *reinterpret_cast<const unsigned int*>(&p));
#else
    *reinterpret_cast<__nv_bfloat162*>(dst + i * N) = p;
#endif
  }
}

// ----------------------------------------------------------------- outlet values
// Sec. 2.3 outflow: for an incoming direction i whose upstream element lies
// beyond the outlet, either extrapolate that element's f_i linearly along -n
// (2 f_i(x - c_i - n) - f_i(x - c_i - 2n); optionally zero-gradient,
// f_i(x - c_i - n)), or, for c_i = -n, correct the pressure:
// f^eq_i(rho0, u) + f^neq_opp(i)(x) with the pre-collision f^neq.
template <int Q, class S>
__global__ void k_outlet(const __grid_constant__ OutletArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  const int64_t k = a.begin + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int lv = 0;
  while (lv < a.nlev && k >= a.lev[lv].end) ++lv;
  if (lv == a.nlev) return;
  const S* __restrict__ src = static_cast<const S*>(a.lev[lv].src);
  const size_t N = (size_t)a.Ntot;
  const int i = a.dir[k];
  R* side = static_cast<R*>(a.side);
  if (a.kind[k] == OUT_EXTRAP) {
    const R fa = Sto<S>::ld(src + (size_t)i * N + a.a[k]);
    side[k] = a.zero_gradient ? fa : R(2) * fa - Sto<S>::ld(src + (size_t)i * N + a.b[k]);
    return;
  }
  if (a.kind[k] == OUT_BOUZIDI) {
    // interpolated bounce-back with the wall at x - q c_i (Sec. 2.3, Bouzidi):
    //   q <  1/2: 2q f*_ib(x) + (1 - 2q) f*_ib(x + c_i)
    //   q >= 1/2: f*_ib(x) / (2q) + (2q - 1) / (2q) f*_i(x)
    // (deviation storage: the weights of each branch sum to one and w_i = w_ib)
    const int ib = opp(i);
    const int64_t e = a.elem[k];
    const double q = a.q ? a.q[k] : 0.5;
    const R fo = Sto<S>::ld(src + (size_t)ib * N + e);
    if (q < 0.5) {
      const int32_t a2 = a.a[k];
      side[k] = a2 < 0 ? fo : R(2.0 * q) * fo + R(1.0 - 2.0 * q) * Sto<S>::ld(src + (size_t)ib * N + a2);
    } else {
      side[k] = R(1.0 / (2.0 * q)) * fo + R((2.0 * q - 1.0) / (2.0 * q)) * Sto<S>::ld(src + (size_t)i * N + e);
    }
    return;
  }
  const int64_t e = a.elem[k];
  R g[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) g[q] = Sto<S>::ld(src + (size_t)q * N + e);
  R F[3] = {R(0), R(0), R(0)};
  if (a.force)
#pragma unroll
    for (int b = 0; b < D; ++b) F[b] = static_cast<const R*>(a.force)[(size_t)b * N + e];
  R rp, j[3];
  raw_moments<Q, R>(g, rp, j);
  const R rho = R(a.rho_off) + rp;
  R u[3] = {R(0), R(0), R(0)};
  R usq = R(0);
#pragma unroll
  for (int b = 0; b < D; ++b) {
    u[b] = (j[b] - R(0.5) * F[b]) / rho;
    usq += u[b] * u[b];
  }
  const int ib = opp(i);
  R gib = R(0);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (q == ib) gib = g[q];
  // f^eq_i(rho0, u) + f^neq_ib, f^neq the pre-collision non-equilibrium part
  // recovered from the stored post-collision pdf: (f* - f^eq - F_ib) / (1 - omega)
  const R om = R(a.lev[lv].omega);
  const R fneq_ib = (gib - geq<Q, R>(ib, rp, rho, u, usq) - guo<Q, R>(ib, om, u, F)) * (R(1) / (R(1) - om));
  const R r0 = R(a.rho0);
  side[k] = geq<Q, R>(i, r0 - R(a.rho_off), r0, u, usq) + fneq_ib;
}

// ----------------------------------------------------------------- GFC source moments
// Interpolation step 1 (Sec. 2.2) as a kernel of its own: density, velocity,
// strain rate and f^neq of the listed sources (elem[k], record rec[k] or k).
// With prev set, the record is the mean of prev and the moments now (the
// source moments at t+1/2 of the linear-in-time mode).  During the steps the
// stream-collide writes the records of the sources it updates (source_out);
// this kernel takes the GhostFromFiner sources after their fill and every
// source when the records have to be rebuilt from a new state.
// The ghost kernels' launch bounds give the block size only, which lets the
// compiler use fewer registers than an explicit minimum of one block.
#ifndef LBM_MOM_BLOCK
#define LBM_MOM_BLOCK 128
#endif
template <class S>
constexpr int kMomBlock = sizeof(S) == 8 ? 32 : LBM_MOM_BLOCK;  // FP64: one warp, as kScBlock
// pdfs of source k (element e): from the state, or as set aside
template <int Q, class S>
__device__ __forceinline__ void load_source(const SavedSources& sv, const S* src, size_t N, int64_t e, int64_t k,
                                            typename Sto<S>::R (&g)[Q]) {
  const S* p = src + e;
  size_t pitch = N;
  if (sv.values) {
    const int32_t i = sv.index[k];
    if (i >= 0) {
      p = static_cast<const S*>(sv.values) + i;
      pitch = (size_t)sv.n;
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) g[q] = Sto<S>::ld(p + q * pitch);
}

template <int Q, class S, bool FORCE>
__global__ void __launch_bounds__(kMomBlock<S>) k_source_moments(const __grid_constant__ MomentsArgs a) {
  using R = typename Sto<S>::R;
  using RL = RecLayout<Q>;
  constexpr int D = Lat<Q>::D;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.nsrc) return;
  const S* __restrict__ src = static_cast<const S*>(a.src);
  const size_t N = (size_t)a.Ntot;
  const int64_t e = a.elem[k];
  const int64_t r = a.rec ? (int64_t)a.rec[k] : k;
  R g[Q];
  load_source<Q, S>(a.saved, src, N, e, k, g);
  R F[3] = {R(0), R(0), R(0)};
  if (FORCE)
#pragma unroll
    for (int b = 0; b < D; ++b) F[b] = static_cast<const R*>(a.force)[(size_t)b * N + e];
  R rec[RL::STRIDE];
  source_record<Q, R, FORCE>(g, pick<R>(a.rx, a.rx32), pick<R>(a.rho_off, a.rho_off32), F, rec);
  if (a.prev) mean_record<Q, R>(static_cast<const R*>(a.prev) + (size_t)r * RL::STRIDE, rec);
  store_record<Q, R>(static_cast<R*>(a.mom) + (size_t)r * RL::STRIDE, rec);
}

// Compact quadratic velocity at the ghost in the octant's local frame, a linear
// map of the sources' local-frame velocities ul and strain rates Sl (see the
// GhostFromCoarser comment below for the closed form).
template <int Q, class R>
__device__ __forceinline__ void compact_uloc(const R (&ul)[4][3], const R (&Sl)[4][Lat<Q>::NS], R (&uloc)[3]) {
  constexpr int D = Lat<Q>::D, NS = Lat<Q>::NS;
  uloc[0] = uloc[1] = uloc[2] = R(0);
  if (D == 3) {
    auto Dx = [&](int c) { return R(0.5) * (-Sl[0][c] + Sl[1][c] + Sl[2][c] - Sl[3][c]); };
    auto Dy = [&](int c) { return R(0.5) * (-Sl[0][c] + Sl[1][c] - Sl[2][c] + Sl[3][c]); };
    auto Dz = [&](int c) { return R(0.5) * (-Sl[0][c] - Sl[1][c] + Sl[2][c] + Sl[3][c]); };
    constexpr int XX = 0, YY = 1, ZZ = 2, XY = 3, YZ = 4, XZ = NS - 1;
    const R h3 = Dz(XY) + Dx(YZ) + Dy(XZ);
    const R sd[3] = {R(0.5) * Dx(XX) + Dy(XY) - R(0.5) * Dx(YY) + Dz(XZ) - R(0.5) * Dx(ZZ),
                     Dx(XY) - R(0.5) * Dy(XX) + R(0.5) * Dy(YY) + Dz(YZ) - R(0.5) * Dy(ZZ),
                     Dx(XZ) - R(0.5) * Dz(XX) + Dy(YZ) - R(0.5) * Dz(YY) + R(0.5) * Dz(ZZ)};
    const R so[3] = {Dy(XX) + Dz(XX) + h3 - R(2) * Dx(YZ), Dx(YY) + Dz(YY) + h3 - R(2) * Dy(XZ),
                     Dx(ZZ) + Dy(ZZ) + h3 - R(2) * Dz(XY)};
#pragma unroll
    for (int b = 0; b < 3; ++b)
      uloc[b] = R(0.625) * ul[0][b] + R(0.125) * (ul[1][b] + ul[2][b] + ul[3][b]) - R(0.1875) * sd[b] -
                R(0.0625) * so[b];
  } else {
    auto Dx = [&](int c) { return R(0.5) * (-Sl[0][c] + Sl[1][c] - Sl[2][c] + Sl[3][c]); };
    auto Dy = [&](int c) { return R(0.5) * (-Sl[0][c] - Sl[1][c] + Sl[2][c] + Sl[3][c]); };
    const R axx = R(0.5) * Dx(0), axy = Dy(0), ayy = Dy(2) - R(0.5) * Dx(1);
    const R bxx = Dx(2) - R(0.5) * Dy(0), byy = R(0.5) * Dy(1), bxy = Dx(1);
    uloc[0] = R(0.5) * ul[0][0] + R(0.25) * (ul[1][0] + ul[2][0]) - R(0.1875) * (axx + ayy) + R(0.0625) * axy;
    uloc[1] = R(0.5) * ul[0][1] + R(0.25) * (ul[1][1] + ul[2][1]) - R(0.1875) * (bxx + byy) + R(0.0625) * bxy;
  }
}

// compact_uloc in FP64 with fewest instructions: the differences' factor 1/2
// in the constants, two of the three differences of a component from the same
// two half differences (3D: 83 instructions for 135).
template <int Q>
__device__ __forceinline__ void compact_uloc64(const double (&ul)[4][3], const double (&Sl)[4][Lat<Q>::NS],
                                               double (&uloc)[3]) {
  constexpr int D = Lat<Q>::D, NS = Lat<Q>::NS;
  double x[NS], y[NS], z[NS];  // twice the differences
#pragma unroll
  for (int c = 0; c < NS; ++c) {
    if (D == 3) {
      const double a = Sl[1][c] - Sl[0][c], b = Sl[2][c] - Sl[3][c];
      x[c] = a + b;
      y[c] = a - b;
      z[c] = (Sl[2][c] + Sl[3][c]) - (Sl[0][c] + Sl[1][c]);
    } else {
      const double a = Sl[1][c] - Sl[0][c], b = Sl[3][c] - Sl[2][c];
      x[c] = b + a;
      y[c] = (Sl[2][c] + Sl[3][c]) - (Sl[0][c] + Sl[1][c]);
      z[c] = 0;
    }
  }
  if (D == 3) {
    constexpr int XX = 0, YY = 1, ZZ = 2, XY = 3, YZ = 4, XZ = NS - 1;
    const double h = z[XY] + x[YZ] + y[XZ];
    const double s1[3] = {x[XX] - x[YY] - x[ZZ], y[YY] - y[XX] - y[ZZ], z[ZZ] - z[XX] - z[YY]};
    const double s2[3] = {y[XY] + z[XZ], x[XY] + z[YZ], x[XZ] + y[YZ]};
    const double s3[3] = {fma(-2.0, x[YZ], y[XX] + z[XX] + h), fma(-2.0, y[XZ], x[YY] + z[YY] + h),
                          fma(-2.0, z[XY], x[ZZ] + y[ZZ] + h)};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const double us = fma(5.0, ul[0][b], ul[1][b]) + (ul[2][b] + ul[3][b]);
      uloc[b] = fma(-0.03125, s3[b], fma(-0.09375, s2[b], fma(-0.046875, s1[b], 0.125 * us)));
    }
  } else {
    uloc[0] = fma(0.03125, y[0], fma(-0.09375, y[2], fma(-0.046875, x[0] - x[1],
                  fma(0.5, ul[0][0], 0.25 * (ul[1][0] + ul[2][0])))));
    uloc[1] = fma(0.03125, x[1], fma(-0.09375, x[2], fma(-0.046875, y[1] - y[0],
                  fma(0.5, ul[0][1], 0.25 * (ul[1][1] + ul[2][1])))));
    uloc[2] = 0;
  }
}

// ----------------------------------------------------------------- GhostFromCoarser
// Interpolation steps 2-5 (Sec. 2.2) for one fine ghost from its four coarse
// sources.  The velocity is the compact quadratic interpolant evaluated at the
// ghost, written in the octant's local frame (signs s_a) in closed form:
// 3D (H, K, M, N at (0,0,0), (1,1,0), (1,0,1), (0,1,1); ghost at (1/4,1/4,1/4)),
//   u_a = 5/8 u_H + 1/8 (u_K + u_M + u_N) - 3/16 (q_xx + q_yy + q_zz)_a
//         - 1/16 (q_xy + q_yz + q_xz)_a,
// with the quadratic coefficients q from the strain-rate differences of
// Eqs. (compact_3D_s); 2D (H, E, N, NE on the unit square, ghost at (1/4,1/4)),
//   u_a = 1/2 u_H + 1/4 (u_E + u_N) - 3/16 (q_xx + q_yy)_a + 1/16 q_xy,a,
// the least-squares linear part over the square.  Density and f^neq are
// linear (weights 5/8,1/8,1/8,1/8 resp. 9/16,3/16,3/16,1/16), f^neq is
// rescaled by omega_c / (m omega_f) (m = dt_c / dt_f), and f = f^eq +
// (1 - omega_f) f^neq is stored as the ghost's post-collision state.  With
// diffusive scaling the velocity and density deviation are converted to the
// fine level's lattice units first, and f^neq's odd part (a flux of order
// tau dt^2 / dx) takes an extra factor 1/2 beside its even part's.
// Ghosts come in groups of 2^d consecutive siblings (the children of one
// coarse parent, octant b = k mod 2^d), and their 4 x 2^d source records are
// 13 distinct ones in 3D (the parent and its 12 edge neighbours), 9 in 2D.  A
// group's lanes stage those records in shared memory with whole-record vector
// loads (one cache line per record), then each lane reads its four sources
// from there.
template <int D>
struct GfcGroup {
  static constexpr int G = 1 << D;           // lanes (siblings) per group
  static constexpr int NSLOT = D == 3 ? 13 : 9;
  // slot of source s (0: parent, 1-3 as in gsrc) for the sibling in octant b
  __device__ static int slot(int s, int b) {
    if (D == 3) return s == 0 ? 0 : s == 1 ? 1 + (b & 3) : s == 2 ? 5 + ((b & 1) | ((b >> 1) & 2)) : 9 + ((b >> 1) & 3);
    return s == 0 ? 0 : s == 1 ? 1 + (b & 1) : s == 2 ? 3 + ((b >> 1) & 1) : 5 + (b & 3);
  }
  // the (source, sibling) pair whose gsrc entry names slot t
  __host__ __device__ static constexpr int src_of(int t) { return t == 0 ? 0 : D == 3 ? 1 + (t - 1) / 4 : (t < 3 ? 1 : t < 5 ? 2 : 3); }
  __host__ __device__ static constexpr int lane_of(int t) {
    return D == 3 ? (t == 0 ? 0 : t < 5 ? t - 1 : t < 9 ? ((t - 5) & 1) | (((t - 5) & 2) << 1) : (t - 9) << 1)
                  : (t == 0 ? 0 : t < 3 ? t - 1 : t < 5 ? (t - 3) << 1 : t - 5);
  }
};

// Interpolation steps 2-5 for ghost k (octant oct) of level L from its group's
// staged records (sg_base: NSLOT padded records), written into L.dst.
template <int Q, class S>
__device__ __forceinline__ void gfc_ghost(const GfcArgs& a, const GfcLevel& L, const typename Sto<S>::R* sg_base, int oct,
                                          int64_t k, bool two) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  using RL = RecLayout<Q>;
  using GG = GfcGroup<LT::D>;
  constexpr int D = LT::D, NS = LT::NS;
  constexpr int PSTR = RL::STRIDE + 4;
  const R* rec[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) rec[s] = sg_base + GG::slot(s, oct) * PSTR;
  R sg[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) sg[c] = ((oct >> c) & 1) ? R(1) : R(-1);
  // local-frame velocity and strain rate of the sources (vector loads of the
  // record tail: rho, u, S)
  R ul[4][3], Sl[4][NS], rps[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    R h[RL::STRIDE - RL::RP];
#pragma unroll
    for (int f = RL::RP; f < RL::STRIDE; f += 4)
      if (f < RL::END) ld4(rec[s] + f, h + (f - RL::RP));
    rps[s] = h[0];
#pragma unroll
    for (int b = 0; b < D; ++b) {
      const R v = h[RL::U - RL::RP + b];
      if constexpr (sizeof(R) == 8) ul[s][b] = flip(v, !((oct >> b) & 1));
      else ul[s][b] = sg[b] * v;
    }
#pragma unroll
    for (int b = 0; b < D; ++b)
#pragma unroll
      for (int c = b; c < D; ++c) {
        const R v = h[RL::SS - RL::RP + sidx<D>(b, c)];
        if constexpr (sizeof(R) == 8) Sl[s][sidx<D>(b, c)] = b == c ? v : flip(v, ((oct >> b) ^ (oct >> c)) & 1);
        else Sl[s][sidx<D>(b, c)] = sg[b] * sg[c] * v;
      }
  }
  R uloc[3];
  if constexpr (sizeof(R) == 8) compact_uloc64<Q>(ul, Sl, uloc);
  else compact_uloc<Q, R>(ul, Sl, uloc);
  R u[3] = {R(0), R(0), R(0)};
  R usq = R(0);
  const auto& un = pick<R>(a.u64, a.u32);
  // FP64 at t + 1/2: the staged records are the sums of the two times';
  // everything taken from them is linear, and the half goes, exactly, into
  // its factors
  [[maybe_unused]] const R half = two ? R(0.5) : R(1);
  R us = un.u_scale;  // to fine lattice units (1 in acoustic scaling)
  if constexpr (sizeof(R) == 8) us *= half;
#pragma unroll
  for (int b = 0; b < D; ++b) {
    u[b] = sg[b] * uloc[b] * us;
    usq += u[b] * u[b];
  }
  const R lw0 = D == 3 ? R(0.625) : R(0.5625);
  const R lw1 = D == 3 ? R(0.125) : R(0.1875);
  const R lw2 = D == 3 ? R(0.125) : R(0.1875);
  const R lw3 = D == 3 ? R(0.125) : R(0.0625);
  R rs = un.r_scale, scale = pick<R>(L.scale, L.scale32);
  if constexpr (sizeof(R) == 8) {
    rs *= half;
    scale *= D == 3 ? 0.125 * half : half;
  }
  const R rp = rs * (lw0 * rps[0] + lw1 * rps[1] + lw2 * rps[2] + lw3 * rps[3]) + un.r_shift;
  const R rho = un.rho_off + rp;
  S* __restrict__ dst = static_cast<S*>(L.dst);
  const size_t N = (size_t)a.Ntot;
  const int64_t e = L.dest0 + k;
  // interpolated f^neq, then f^eq per pair of opposite velocities (shared even part)
  R fn[Q];
#pragma unroll
  for (int q0 = 0; q0 < Q; q0 += 4) {
    R f0[4], f1[4], f2[4], f3[4];
    ld4(rec[0] + RL::FN + q0, f0);
    ld4(rec[1] + RL::FN + q0, f1);
    ld4(rec[2] + RL::FN + q0, f2);
    ld4(rec[3] + RL::FN + q0, f3);
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (q0 + c < Q) {
        // FP64, 3D: 8 times the interpolated value, in three instructions
        if constexpr (sizeof(R) == 8 && D == 3) fn[q0 + c] = fma(5.0, f0[c], f1[c]) + (f2[c] + f3[c]);
        else fn[q0 + c] = lw0 * f0[c] + lw1 * f1[c] + lw2 * f2[c] + lw3 * f3[c];
      }
  }
  const R base = rp - R(1.5) * rho * usq;
  dst[e] = Sto<S>::cv(R(LT::w(0)) * base + scale * fn[0]);
  // diffusive scaling: f^neq's odd part takes an extra factor (odd_ratio)
  const bool odd_rescale = a.odd_rescale != 0;
  const R ro = un.odd;
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    R cu = R(0);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      if (LT::c(i, b) > 0) cu += u[b];
      if (LT::c(i, b) < 0) cu -= u[b];
    }
    if constexpr (sizeof(R) == 8) {
      double fa = fn[i], fb = fn[i + 1];
      if (odd_rescale) {
        const double fe = 0.5 * (fa + fb), fo = 0.5 * (fa - fb) * ro;
        fa = fe + fo;
        fb = fe - fo;
      }
      // the products with a weight are shared by all its directions
      const double w = LT::w(i), wr = 3.0 * w * rho, even = fma((4.5 * w * rho) * cu, cu, w * base);
      dst[(size_t)i * N + e] = fma(scale, fa, fma(wr, cu, even));
      dst[(size_t)(i + 1) * N + e] = fma(scale, fb, fma(-wr, cu, even));
      continue;
    }
    const R w = R(LT::w(i));
    const R even = w * (base + R(4.5) * rho * cu * cu);
    const R odd = w * R(3) * rho * cu;
    R fa = fn[i], fb = fn[i + 1];
    if (odd_rescale) {
      const R fe = R(0.5) * (fa + fb), fo = R(0.5) * (fa - fb) * ro;
      fa = fe + fo;
      fb = fe - fo;
    }
    dst[(size_t)i * N + e] = Sto<S>::cv(even + odd + scale * fa);
    dst[(size_t)(i + 1) * N + e] = Sto<S>::cv(even - odd + scale * fb);
  }
}


#ifndef LBM_GFC_BLOCK
#define LBM_GFC_BLOCK 64
#endif
template <class S>
constexpr int kGfcBlock = sizeof(S) == 8 ? 32 : LBM_GFC_BLOCK;  // FP64: one warp, as kScBlock
// ONE: a single level, all of it at t + 1/2.
template <int Q, class S, bool TWO, bool ONE = false>
__global__ void __launch_bounds__(kGfcBlock<S>) k_fill_gfc(const __grid_constant__ GfcArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  using RL = RecLayout<Q>;
  using GG = GfcGroup<LT::D>;
  constexpr int G = GG::G, NSLOT = GG::NSLOT;
  constexpr int PSTR = RL::STRIDE + 4;  // padded record: sibling lanes' reads fall in distinct banks
  constexpr int NGRP = kGfcBlock<S> / G;
  __shared__ __align__(16) R stage[NGRP * NSLOT * PSTR];
  const int seg = ONE ? 0 : segment_of(a.first, a.nseg, blockIdx.x);
  const GfcLevel& L = a.lev[seg];
  const int64_t k = (int64_t)(blockIdx.x - (ONE ? 0u : a.first[seg])) * kGfcBlock<S> + threadIdx.x;
  const int oct = threadIdx.x & (G - 1);  // octant of the ghost
  const int grp = threadIdx.x / G;
  const bool active = k < L.ng;                   // ng is a multiple of G: whole groups
  const unsigned lane0 = (threadIdx.x & 31) & ~(unsigned)(G - 1);
  int32_t src[4] = {0, 0, 0, 0};
  if (active)
#pragma unroll
    for (int s = 0; s < 4; ++s) src[s] = L.gsrc[(size_t)s * L.ng + k];
  const R* __restrict__ mom = static_cast<const R*>(L.mom);
  const R* __restrict__ mom2 = static_cast<const R*>(L.mom2);
  const bool two = ONE || mom2 != nullptr;
  R* sg_base = stage + grp * NSLOT * PSTR;
  wait_for_previous();
  // every record's loads are issued before the first is stored, so that they
  // overlap (one round trip instead of one per record).  At t + 1/2 in two
  // batches where levels share the launch (sphere of 8.6e7 elements: 146
  // against 153 us) and in one where a level is alone (99 against 113 us).
  constexpr int CH = RL::STRIDE / 4 / G > 0 ? (RL::STRIDE / 4 + G - 1) / G : 1;  // vectors per lane and record
  constexpr int BATCH = sizeof(R) == 8 ? (NSLOT * CH > 16 ? 5 : 7) : TWO && !(ONE && CH == 1) ? (NSLOT + 1) / 2 : NSLOT;
#pragma unroll
  for (int t0 = 0; t0 < NSLOT; t0 += BATCH) {
    R v[BATCH][CH][4];
    int r[BATCH];
#pragma unroll
    for (int t = t0; t < t0 + BATCH && t < NSLOT; ++t) {
      r[t - t0] = __shfl_sync(0xffffffffu, src[GG::src_of(t)], lane0 + GG::lane_of(t));
#pragma unroll
      for (int c = 0; c < CH; ++c)
        if (active && oct + c * G < RL::STRIDE / 4)
          ld4(mom + (size_t)r[t - t0] * RL::STRIDE + 4 * (oct + c * G), v[t - t0][c]);
    }
    if (TWO && two) {
      // the records at t + 1/2: the means of those at t and t + 1 (FP64: the
      // sums, gfc_ghost takes the half)
      R w[BATCH][CH][4];
#pragma unroll
      for (int t = t0; t < t0 + BATCH && t < NSLOT; ++t)
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (active && oct + c * G < RL::STRIDE / 4)
            ld4(mom2 + (size_t)r[t - t0] * RL::STRIDE + 4 * (oct + c * G), w[t - t0][c]);
#pragma unroll
      for (int t = t0; t < t0 + BATCH && t < NSLOT; ++t)
#pragma unroll
        for (int c = 0; c < CH; ++c)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            v[t - t0][c][j] = sizeof(R) == 8 ? v[t - t0][c][j] + w[t - t0][c][j] : R(0.5) * (v[t - t0][c][j] + w[t - t0][c][j]);
    }
#pragma unroll
    for (int t = t0; t < t0 + BATCH && t < NSLOT; ++t)
#pragma unroll
      for (int c = 0; c < CH; ++c)
        if (active && oct + c * G < RL::STRIDE / 4) st4(sg_base + t * PSTR + 4 * (oct + c * G), v[t - t0][c]);
  }
  __syncwarp();
  let_next_start();
  // outer-layer ghosts are staged with their group but, when skipped, not written
  if (!active || (L.skip_outer && (L.oct[k] & kGfcOuter))) return;
  gfc_ghost<Q, S>(a, L, sg_base, oct, k, TWO && two);
}

// ----------------------------------------------------------------- GhostFromFiner
// Coarse ghost from its 2^d children (Sec. 2.2 steps 1-5 with the children as
// sources; they surround the ghost symmetrically at +-1/4 coarse cell).
// Density and f^neq: the children's mean.  Velocity: the children's mean minus
// (1/32) lap u, with lap u_a = 2 d_c S_ac - d_a S_cc from the children's strain
// rates (differences across the children's cube).  f^neq is rescaled by
// m omega_f / omega_c (m = dt_c / dt_f); f = f^eq + (1 - omega_c) f^neq.  With
// diffusive scaling the mean velocity and density deviation are converted to
// the coarse level's lattice units, and f^neq's odd part takes an extra
// factor 2.
// One group of 2^d consecutive lanes per ghost: lane b loads child b (siblings
// are contiguous, so the group's loads are coalesced), and the sums over the
// children are shuffles inside the group.
// Ghosts that are GhostFromCoarser sources also get their record here (step 1
// of Sec. 2.2 for the next finer level): the group stages the values as
// stored in shared memory and one thread per ghost forms the record, the same
// arithmetic as k_source_moments, one launch fewer between a level's
// GhostFromFiner and GhostFromCoarser fills.
template <class S>
constexpr int kGffBlock = sizeof(S) == 8 ? 64 : 256;  // FP64: small blocks, as kScBlock
template <int Q, class S, bool FORCE>
__global__ void __launch_bounds__(kGffBlock<S>) k_fill_gff(const __grid_constant__ GffArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  using RL = RecLayout<Q>;
  constexpr int D = LT::D, NS = LT::NS, NCH = 1 << D, GPB = kGffBlock<S> / NCH;
  __shared__ R stored[Q][GPB + 1];
  const int seg = segment_of(a.first, a.nseg, blockIdx.x);
  const GffLevel& L = a.lev[seg];
  const auto& un = pick<R>(a.u64, a.u32);
  const int64_t t = (int64_t)(blockIdx.x - a.first[seg]) * kGffBlock<S> + threadIdx.x;
  const int64_t k = t / NCH;
  const int b = (int)(t % NCH);
  const bool active = k < L.ng;
  const S* __restrict__ src = static_cast<const S*>(L.src_fine);
  const size_t N = (size_t)a.Ntot;
  const R rho_off = un.rho_off;
  R rp = R(0), u[3] = {R(0), R(0), R(0)}, fneq[Q], Sv[NS];
#pragma unroll
  for (int q = 0; q < Q; ++q) fneq[q] = R(0);
#pragma unroll
  for (int s = 0; s < NS; ++s) Sv[s] = R(0);
  const int64_t child = active ? (int64_t)L.child0[k] + b : 0;
  wait_for_previous();
  if (active) {
    const int64_t e = child;
    R g[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) g[q] = Sto<S>::ld(src + (size_t)q * N + e);
    R F[3] = {R(0), R(0), R(0)};
    if (FORCE)
#pragma unroll
      for (int c = 0; c < D; ++c) F[c] = static_cast<const R*>(a.force)[(size_t)c * N + e];
    if constexpr (sizeof(R) == 8) post_moments64<Q, FORCE>(g, a.rx_f64[seg], rho_off, F, rp, u, fneq, Sv);
    else post_moments<Q, R, true, FORCE>(g, L.rx_f.omega, L.rx_f.r1w, rho_off, F, rp, u, fneq, Sv);
    if (a.odd_rescale) {
      // diffusive scaling: f^neq's odd part takes an extra factor (the sum
      // over the children is linear, so each child's share is rescaled)
      const R ro = un.odd;
#pragma unroll
      for (int i = 1; i < Q; i += 2) {
        const R fe = R(0.5) * (fneq[i] + fneq[i + 1]), fo = R(0.5) * (fneq[i] - fneq[i + 1]) * ro;
        fneq[i] = fe + fo;
        fneq[i + 1] = fe - fo;
      }
    }
  }
  let_next_start();
  // The ghost's velocity, mean minus (1/32) lap u, is linear in the children's
  // values, and so is lap u_a = dfac sum_c (2 d_c S_ac - d_a S_cc) with d_c the
  // difference across the cube (+ for children with bit c set, - otherwise):
  // each lane forms its child's share and the group sums d + 1 values.
  // d_c S (coarse units): S_coarse = m S_fine (m = dt_c / dt_f); difference of
  // the two half-cubes over a distance of 1/2 coarse cell -> factor m 2^{2-D}.
  // The mean velocity goes to coarse units with u_scale (a power of two, so
  // inv_u is exact).
  const R inv = R(1) / R(NCH);
  const R inv_u = inv * un.u_scale;
  const R dfac = un.tratio * R(D == 3 ? 0.5 : 1.0);
  R rpm = rp * inv, uP[3] = {R(0), R(0), R(0)};
  if constexpr (sizeof(R) == 8) {
    double tr = 0;
#pragma unroll
    for (int c = 0; c < D; ++c) tr += Sv[c];
#pragma unroll
    for (int aa = 0; aa < D; ++aa) {
      double s2 = 0;
#pragma unroll
      for (int c = 0; c < D; ++c) s2 += flip(Sv[sidx<D>(aa, c)], !((b >> c) & 1));
      const double lap = fma(2.0, s2, flip(tr, (b >> aa) & 1));
      uP[aa] = fma(-dfac / 32.0, lap, u[aa] * inv_u);
    }
  } else {
#pragma unroll
    for (int aa = 0; aa < D; ++aa) {
      const R sa = ((b >> aa) & 1) ? R(1) : R(-1);
      R lap = R(0);
#pragma unroll
      for (int c = 0; c < D; ++c) {
        const R sc = ((b >> c) & 1) ? R(1) : R(-1);
        lap += dfac * (R(2) * sc * Sv[sidx<D>(aa, c)] - sa * Sv[sidx<D>(c, c)]);
      }
      uP[aa] = u[aa] * inv_u - lap * R(1.0 / 32.0);
    }
  }
#pragma unroll
  for (int o = 1; o < NCH; o <<= 1) {
    rpm += __shfl_xor_sync(0xffffffffu, rpm, o);
#pragma unroll
    for (int c = 0; c < D; ++c) uP[c] += __shfl_xor_sync(0xffffffffu, uP[c], o);
  }
  // f^neq: reduce-scatter (recursive halving), lane b ends with the sums for
  // q = j 2^d + b; at half-width h a lane keeps the half of its columns on its
  // side of bit h and receives its partner's partial sums of that half
  constexpr int NR = (Q + NCH - 1) / NCH;
  R W[NR][NCH];
#pragma unroll
  for (int j = 0; j < NR; ++j)
#pragma unroll
    for (int c = 0; c < NCH; ++c) W[j][c] = j * NCH + c < Q ? fneq[j * NCH + c] : R(0);
#pragma unroll
  for (int h = NCH / 2; h >= 1; h >>= 1) {
    const bool hi = (b & h) != 0;
#pragma unroll
    for (int j = 0; j < NR; ++j)
#pragma unroll
      for (int c = 0; c < h; ++c) {
        const R send = hi ? W[j][c] : W[j][c + h];
        const R keep = hi ? W[j][c + h] : W[j][c];
        W[j][c] = keep + __shfl_xor_sync(0xffffffffu, send, h);
      }
  }
  const int64_t e = k < L.n_inner ? L.dest0 + k : L.dest_outer + (k - L.n_inner);
  if (active) {
    R usq = R(0);
#pragma unroll
    for (int aa = 0; aa < D; ++aa) usq += uP[aa] * uP[aa];
    rpm = un.r_scale * rpm + un.r_shift;  // to coarse units (unchanged in acoustic scaling)
    const R rho = rho_off + rpm;
    const R scale = pick<R>(a.scale[seg], L.scale32);
    S* __restrict__ dst = static_cast<S*>(L.dst);
    // the group's lanes share the Q stores: lane b the directions j 2^d + b,
    // whose c_i it looks up at run time (a compile-time loop over all Q would
    // issue every direction's arithmetic in every lane)
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      const int q = j * NCH + b;
      if (q < Q) {
        R cu = R(0);
#pragma unroll
        for (int aa = 0; aa < D; ++aa) cu += R(LatRt<Q>::c(q, aa)) * uP[aa];
        const R feq = LatRt<Q>::template w<R>(q) * (rpm + rho * (R(3) * cu + R(4.5) * cu * cu - R(1.5) * usq));
        const S v = Sto<S>::cv(feq + scale * W[j][0]);
        dst[(size_t)q * N + e] = v;
        stored[q][threadIdx.x / NCH] = Sto<S>::ld(&v);
      }
    }
  }
  if (!L.rec_out) return;  // uniform over the block
  __syncthreads();
  const int64_t kr = (int64_t)(blockIdx.x - a.first[seg]) * GPB + threadIdx.x;
  if (threadIdx.x >= GPB || kr >= L.ng) return;
  const int64_t er = kr < L.n_inner ? L.dest0 + kr : L.dest_outer + (kr - L.n_inner);
  const int64_t r = source_index(a.sources, er);
  if (r < 0) return;
  R g[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) g[q] = stored[q][threadIdx.x];
  R F[3] = {R(0), R(0), R(0)};
  if (FORCE)
#pragma unroll
    for (int c = 0; c < D; ++c) F[c] = static_cast<const R*>(a.force)[(size_t)c * N + er];
  R rec[RL::STRIDE];
  source_record<Q, R, FORCE>(g, pick<R>(a.rx_c64[seg], a.rx_c[seg]), rho_off, F, rec);
  store_record<Q, R>(static_cast<R*>(L.rec_out) + r * RL::STRIDE, rec);
}

// ----------------------------------------------------------------- set-up (compute type) / output (FP64)
template <int Q, class S>
__global__ void k_fill_rest(const FillArgs a) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.Ntot) return;
  S* p = static_cast<S*>(a.pdf);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    p[(size_t)q * a.Ntot + e] = Sto<S>::cv(typename Sto<S>::R(Lat<Q>::w(q) * (a.rho0 - a.rho_off)));
}

// Initial state, Sec. 4.1: f = f^eq + (1 - omega) f^neq + df with
// f^neq_i = -(3 w_i rho / omega) (c_i c_i - I/3) : S.  HAS_S: a strain rate is
// given (a template flag, so that the loop over the directions has no branch
// on it and unrolls into compile-time lattice constants).
template <int Q, class S, bool HAS_S>
__global__ void k_init(const InitArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  constexpr int D = LT::D, NS = LT::NS;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.cnt) return;
  const int64_t k = a.first + t;
  const int li = a.ulev[k];
  // equilibrium in the deviation form of the storage (g = f - w rho_off),
  // computed in the storage's compute type like the collision's equilibrium
  const R rho = R(a.rho[t]);
  const R rp = R(a.rho[t] - a.rho_off);
  R u[3] = {R(0), R(0), R(0)}, usq = R(0);
#pragma unroll
  for (int b = 0; b < D; ++b) {
    u[b] = R(a.u[t * D + b]);
    usq += u[b] * u[b];
  }
  R sv[NS], tr = R(0);
  if (HAS_S) {
#pragma unroll
    for (int j = 0; j < NS; ++j) sv[j] = R(a.S[t * NS + j]);
#pragma unroll
    for (int b = 0; b < D; ++b) tr += sv[sidx<D>(b, b)];
  }
  const double* df = a.df ? a.df + t * Q : nullptr;
  const R om = R(a.omega[li]);
  S* out = static_cast<S*>(a.temp) + k;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    R g = geq<Q, R>(q, rp, rho, u, usq);
    if (HAS_S) {
      R qs = R(0);
#pragma unroll
      for (int b = 0; b < D; ++b)
#pragma unroll
        for (int c = b; c < D; ++c) qs += R((b == c ? 1 : 2) * LT::c(q, b) * LT::c(q, c)) * sv[sidx<D>(b, c)];
      // post-collision non-equilibrium part (1 - omega) f^neq of the strain rate
      g += (R(1) - om) * (-(R(3.0 * LT::w(q)) * rho / om) * (qs - tr / R(3)));
    }
    if (df) g += R(df[q]);
    out[(size_t)q * a.n_user] = Sto<S>::cv(g);
  }
}

// caller-ordered initial pdfs -> element slots (coalesced writes in slot order)
template <int Q, class S>
__global__ void k_init_place(const PlaceArgs a) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.Ntot) return;
  const int32_t u = a.slot_user[e];
  if (u < 0) return;
  const S* src = static_cast<const S*>(a.temp) + u;
  S* dst = static_cast<S*>(a.dst) + e;
#pragma unroll
  for (int q = 0; q < Q; ++q) dst[(size_t)q * a.Ntot] = src[(size_t)q * a.n_user];
}

// Moments or pdfs of a chunk of caller-order elements, in FP64 whatever the
// storage.  The moments are bound by the FP64 pipe: without a force the
// forcing terms are left out at compile time, and post_moments64 takes a third
// of the instructions of the general form (1.31e5 D3Q19 elements: 19 us; the
// general form took 0.6 ms per 1.05e6 elements, more than their copy).
template <int Q, class S, bool FORCE>
__global__ void __launch_bounds__(128) k_out(const __grid_constant__ OutArgs a) {
  using R = typename Sto<S>::R;
  using LT = Lat<Q>;
  constexpr int D = LT::D, NS = LT::NS;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.cnt) return;
  const int64_t k = a.first + t;
  const int li = a.ulev[k];
  const S* cur = static_cast<const S*>(((a.parity >> li) & 1) ? a.B : a.A);
  const int64_t e = a.uslot[k];
  R gs[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) gs[q] = Sto<S>::ld(cur + (size_t)q * a.Ntot + e);
  double g[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) g[q] = (double)gs[q];
  if (a.f) {
    double* o = a.f + t * Q;
#pragma unroll
    for (int q = 0; q < Q; ++q) o[q] = g[q] + LT::w(q) * a.rho_off;
  }
  if (!a.rho && !a.u && !a.S) return;
  double F[3] = {0, 0, 0};
  if (FORCE)
#pragma unroll
    for (int b = 0; b < D; ++b) F[b] = (double)static_cast<const R*>(a.force)[(size_t)b * a.Ntot + e];
  double rp, u[3], fneq[Q], Sv[NS];
  post_moments64<Q, FORCE>(g, a.rx[li], a.rho_off, F, rp, u, fneq, Sv);
  if (a.rho) a.rho[t] = a.rho_off + rp;
  if (a.u)
#pragma unroll
    for (int b = 0; b < D; ++b) a.u[t * D + b] = u[b];
  if (a.S)
#pragma unroll
    for (int s = 0; s < NS; ++s) a.S[t * NS + s] = Sv[s];
}

template <int Q, class S>
__global__ void k_set_state(const SetStateArgs a) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.cnt) return;
  const int64_t k = a.first + t;
  const int li = a.ulev[k];
  S* cur = static_cast<S*>(((a.parity >> li) & 1) ? a.B : a.A);
  const int64_t e = a.uslot[k];
#pragma unroll
  for (int q = 0; q < Q; ++q)
    cur[(size_t)q * a.Ntot + e] =
        Sto<S>::cv(typename Sto<S>::R(a.f[t * Q + q] - Lat<Q>::w(q) * a.rho_off));
}

template <int Q, class S>
__global__ void k_gather_ghosts(const GatherGhostArgs a) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.cnt) return;
  const S* p = static_cast<const S*>(a.pdf);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    a.stage[t * Q + q] = (double)Sto<S>::ld(p + (size_t)q * a.Ntot + a.first_global + t) + Lat<Q>::w(q) * a.rho_off;
}

// ----------------------------------------------------------------- FP64 reductions
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block sums of the threads' values v[0..NV) where bit k of `used` is set
// (uniform), out[k] = 0 elsewhere: one warp per value, NV (threads / 32 + 5)
// FP64 instructions a block (in every warp: 4 times as many, on the narrow
// FP64 pipe, 11 us for a launch of 512 blocks of 256 threads).
template <int NV, int BLOCK>
__device__ __forceinline__ void block_sum_store(const double (&v)[NV], double* out, unsigned used) {
  __shared__ double sh[NV][BLOCK];
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if ((used >> k) & 1u) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int k = threadIdx.x >> 5; k < NV; k += BLOCK / 32) {
    double s = 0.0;
    if ((used >> k) & 1u) {
#pragma unroll
      for (int t = 0; t < BLOCK; t += 32) s += sh[k][t + lane];
      s = warp_sum(s);
    }
    if (lane == 0) out[k] = s;
  }
}

// Running sum of FP32 values kept as an unevaluated pair hi + lo (Knuth's
// two-sum: hi + x is split exactly into its rounded value and the rounding
// error, which lo collects): about twice the FP32 precision on the FP32
// pipe, converted to FP64 once at the end.
struct SumF2 {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = hi + x;
    const float bp = s - hi;
    lo += (hi - (s - bp)) + (x - bp);
    hi = s;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// mass, momentum, obstacle force (momentum exchange, Sec. 2.3) and kinetic energy
// of all levels; one partial row per block, grid fixed by the mesh ->
// deterministic order.  One launch with blocks for the elements there are (one
// of 512 blocks per level before: 50 us of kernels for the four-level D2Q9
// cylinder, where the blocks' sums alone bound it).
// A thread sums its elements' moments (FP32 compute type: as two-float sums,
// which keeps the FP64 pipe, GB300's narrow one, out of the per-element work;
// FP64 storage: in FP64), then the block and grid sums are FP64.
template <class S>
constexpr int kRedBlock = sizeof(S) == 8 ? 128 : 256;
template <int Q, class S>
__global__ void __launch_bounds__(kRedBlock<S>) k_reduce(const __grid_constant__ ReduceArgs a) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  const int seg = segment_of(a.first, a.nseg, blockIdx.x);
  const ReduceLevel& L = a.lev[seg];
  const unsigned blocks = (seg + 1 < a.nseg ? a.first[seg + 1] : gridDim.x) - a.first[seg];
  const int64_t t0 = (int64_t)(blockIdx.x - a.first[seg]) * kRedBlock<S> + threadIdx.x;
  const S* p = static_cast<const S*>(L.pdf);
  const size_t N = (size_t)a.Ntot;
  const int64_t stride = (int64_t)blocks * kRedBlock<S>;
  // each element's moments in the storage's compute type (the sums of its Q
  // stored values); the accumulation over elements in FP64
  // (the level volume and rho_off are applied once per thread below)
  using R = typename Sto<S>::R;
  constexpr bool F2 = sizeof(R) == 4;
  SumF2 sf[5];  // rp, rho u, kinetic energy (FP32 compute type)
  int64_t cnt = 0;
  for (int64_t e = L.begin + t0; e < L.end; e += stride) {
    R g[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) g[q] = Sto<S>::ld(p + (size_t)q * N + e);
    R rp, j[3];
    if constexpr (F2) raw_moments<Q, R>(g, rp, j);
    else raw_moments64<Q>(g, rp, j);
    R F[3] = {R(0), R(0), R(0)};
    if (a.force)
      for (int b = 0; b < D; ++b) F[b] = static_cast<const R*>(a.force)[(size_t)b * N + e];
    const R rho = R(a.rho_off) + rp;
    R uu = R(0);
    R m[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int b = 0; b < D; ++b) {
      m[b] = j[b] - R(0.5) * F[b];  // rho u
      uu += m[b] * m[b];
    }
    const R ke = R(0.5) * uu / rho;
    if constexpr (F2) {
      sf[0].add(rp);
#pragma unroll
      for (int b = 0; b < D; ++b) sf[1 + b].add(m[b]);
      sf[4].add(ke);
    } else {
      acc[0] += (double)rp;
#pragma unroll
      for (int b = 0; b < D; ++b) acc[1 + b] += (double)m[b];
      acc[7] += (double)ke;
    }
    ++cnt;
  }
  if constexpr (F2) {
    acc[0] = sf[0].value();
#pragma unroll
    for (int b = 0; b < 3; ++b) acc[1 + b] = sf[1 + b].value();
    acc[7] = sf[4].value();
  }
  if (L.r_scale == 1.0)
    acc[0] = L.vol * (acc[0] + (double)cnt * a.rho_off);
  else  // density deviations in another level's units
    acc[0] = L.vol * ((double)cnt * a.rho0 + L.r_scale * (acc[0] + (double)cnt * (a.rho_off - a.rho0)));
#pragma unroll
  for (int b = 0; b < 3; ++b) acc[1 + b] *= L.vol_m;
  acc[7] *= L.vol_k;
  // momentum exchange (Sec. 2.3): the link carries c_ib (f*_ib(x) + f_i(x)) to
  // the body, f_i the bounce-back value of the next step (interpolated with
  // the wall distance q; q = 1/2 gives 2 c_ib f*_ib)
  for (int64_t l = t0; l < L.obs_n; l += stride) {
    const int i = L.obs_dir[l];
    const int ib = opp(i);
    const int64_t e = L.obs_elem[l];
    const double q = L.obs_q ? L.obs_q[l] : 0.5;
    const double go = (double)Sto<S>::ld(p + (size_t)ib * N + e);
    double gb;
    if (q < 0.5) {
      const int32_t a2 = L.obs_a ? L.obs_a[l] : -1;
      gb = a2 < 0 ? go : 2.0 * q * go + (1.0 - 2.0 * q) * (double)Sto<S>::ld(p + (size_t)ib * N + a2);
    } else {
      gb = go / (2.0 * q) + (2.0 * q - 1.0) / (2.0 * q) * (double)Sto<S>::ld(p + (size_t)i * N + e);
    }
    const double sum = go + gb + 2.0 * LT::w(ib) * a.rho_off;
#pragma unroll
    for (int b = 0; b < D; ++b) acc[4 + b] += L.fscale * LT::c(ib, b) * sum;
  }
  // mass, kinetic energy, momentum, and forces where there are obstacle links
  const unsigned axes = (1u << D) - 1u;
  block_sum_store<8, kRedBlock<S>>(acc, a.partial + (size_t)blockIdx.x * 8,
                                   0x81u | axes << 1 | (L.obs_n > 0 ? axes << 4 : 0u));
}

// ----------------------------------------------------------------- launchers
inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Calls f with std::integral_constant<int, Q> for the run-time stencil Q
// (9, 19 or 27; the mesh builder rejects anything else).
template <class F>
inline void with_q(int Q, F&& f) {
  if (Q == 9) f(std::integral_constant<int, 9>{});
  else if (Q == 19) f(std::integral_constant<int, 19>{});
  else f(std::integral_constant<int, 27>{});
}

// Launches kernel(a), as a programmatic dependent of the stream's previous
// kernel where a.chain says so.
template <class Args>
inline void launch(void (*kernel)(const Args), unsigned grid, int block, cudaStream_t st, const Args& a) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = a.chain ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, a);
}

template <class S>
struct Launch {
  // first blocks of the segments, in order, from the threads each needs;
  // returns the grid
  template <class Args, class Work>
  static unsigned assign_blocks(Args& a, int block, Work&& threads) {
    unsigned at = 0;
    for (int k = 0; k < a.nseg; ++k) {
      a.first[k] = at;
      at += blocks_for(threads(k), block);
    }
    return at;
  }
  static bool any_records(const ScArgs& a) {
    for (int k = 0; k < a.nseg; ++k)
      if (a.seg[k].rec_out) return true;
    return false;
  }
  static int sc_interior(int Q, bool force, ScArgs& a, cudaStream_t st) {
    const bool moms = any_records(a);
    int n = 0;
    with_q(Q, [&](auto q) {
      constexpr int QQ = decltype(q)::value;
      if constexpr (std::is_same<S, __nv_bfloat16>::value) {
        // BF16: two elements per thread, one brick per warp (on levels without
        // GFC sources; the others take the one-element kernel with its record
        // epilogue)
        if (!moms) {
          ScArgs one = a;
          one.nseg = 1;
          for (int k = 0; k < a.nseg; ++k) {
            one.seg[0] = a.seg[k];
            const unsigned g = blocks_for(32ll * a.seg[k].n, LBM_BR_PAIR_BLOCK);
            if (force) launch(k_sc_interior_pair<QQ, true>, g, LBM_BR_PAIR_BLOCK, st, one);
            else launch(k_sc_interior_pair<QQ, false>, g, LBM_BR_PAIR_BLOCK, st, one);
          }
          n = a.nseg;
          return;
        }
      }
      const unsigned g = assign_blocks(a, kScBlock<S>, [&](int k) { return 64ll * a.seg[k].n; });
      if (!g) return;
      n = 1;
      if (force) {
        if (moms) launch(k_sc_interior<QQ, S, true, true>, g, kScBlock<S>, st, a);
        else launch(k_sc_interior<QQ, S, true, false>, g, kScBlock<S>, st, a);
      } else {
        if (moms) launch(k_sc_interior<QQ, S, false, true>, g, kScBlock<S>, st, a);
        else launch(k_sc_interior<QQ, S, false, false>, g, kScBlock<S>, st, a);
      }
    });
    return n;
  }
  static int sc_rest(int Q, bool force, ScArgs& a, cudaStream_t st) {
    const bool moms = any_records(a);
    const unsigned g =
        assign_blocks(a, kScBlock<S>, [&](int k) { return (a.seg[k].list ? 1ll : 64ll) * a.seg[k].n; });
    if (!g) return 0;
    bool list = false;
    for (int k = 0; k < a.nseg; ++k) list |= a.seg[k].list != 0;
    with_q(Q, [&](auto q) {
      auto go = [&](auto F, auto M, auto L) {
        launch(k_sc_rest<decltype(q)::value, S, decltype(F)::value, decltype(M)::value, decltype(L)::value>, g,
               kScBlock<S>, st, a);
      };
      using T = std::true_type;
      using U = std::false_type;
      auto by_list = [&](auto F, auto M) { list ? go(F, M, T{}) : go(F, M, U{}); };
      if (force) moms ? by_list(T{}, T{}) : by_list(T{}, U{});
      else moms ? by_list(U{}, T{}) : by_list(U{}, U{});
    });
    return 1;
  }
  static int outlet(int Q, const OutletArgs& a, cudaStream_t st) {
    if (!a.nlev) return 0;
    const int64_t n = a.lev[a.nlev - 1].end - a.begin;
    with_q(Q, [&](auto q) { k_outlet<decltype(q)::value, S><<<blocks_for(n, kMomBlock<S>), kMomBlock<S>, 0, st>>>(a); });
    return 1;
  }
  static int source_moments(int Q, const MomentsArgs& a, cudaStream_t st) {
    if (a.nsrc <= 0) return 0;
    with_q(Q, [&](auto q) {
      constexpr int QQ = decltype(q)::value;
      const unsigned g = blocks_for(a.nsrc, kMomBlock<S>);
      if (a.force) k_source_moments<QQ, S, true><<<g, kMomBlock<S>, 0, st>>>(a);
      else k_source_moments<QQ, S, false><<<g, kMomBlock<S>, 0, st>>>(a);
    });
    return 1;
  }
  static int fill_gfc(int Q, GfcArgs& a, cudaStream_t st) {
    const unsigned g = assign_blocks(a, kGfcBlock<S>, [&](int k) { return (int64_t)a.lev[k].ng; });
    if (!g) return 0;
    bool two = false;
    for (int k = 0; k < a.nseg; ++k) two |= a.lev[k].mom2 != nullptr;
    with_q(Q, [&](auto q) {
      if (two && a.nseg == 1) launch(k_fill_gfc<decltype(q)::value, S, true, true>, g, kGfcBlock<S>, st, a);
      else if (two) launch(k_fill_gfc<decltype(q)::value, S, true>, g, kGfcBlock<S>, st, a);
      else launch(k_fill_gfc<decltype(q)::value, S, false>, g, kGfcBlock<S>, st, a);
    });
    return 1;
  }
  static int fill_gff(int Q, GffArgs& a, cudaStream_t st) {
    int n = 0;
    with_q(Q, [&](auto q) {
      constexpr int QQ = decltype(q)::value;
      const unsigned g =
          assign_blocks(a, kGffBlock<S>, [&](int k) { return (int64_t)a.lev[k].ng << Lat<QQ>::D; });
      if (!g) return;
      n = 1;
      if (a.force) launch(k_fill_gff<QQ, S, true>, g, kGffBlock<S>, st, a);
      else launch(k_fill_gff<QQ, S, false>, g, kGffBlock<S>, st, a);
    });
    return n;
  }
  static void fill_rest(int Q, const FillArgs& a, cudaStream_t st) {
    with_q(Q, [&](auto q) { k_fill_rest<decltype(q)::value, S><<<blocks_for(a.Ntot, 256), 256, 0, st>>>(a); });
  }
  static void init(int Q, const InitArgs& a, cudaStream_t st) {
    if (a.cnt <= 0) return;
    with_q(Q, [&](auto q) {
      if (a.S) k_init<decltype(q)::value, S, true><<<blocks_for(a.cnt, 128), 128, 0, st>>>(a);
      else k_init<decltype(q)::value, S, false><<<blocks_for(a.cnt, 128), 128, 0, st>>>(a);
    });
  }
  static void init_place(int Q, const PlaceArgs& a, cudaStream_t st) {
    with_q(Q, [&](auto q) { k_init_place<decltype(q)::value, S><<<blocks_for(a.Ntot, 256), 256, 0, st>>>(a); });
  }
  static void out(int Q, const OutArgs& a, cudaStream_t st) {
    if (a.cnt <= 0) return;
    with_q(Q, [&](auto q) {
      constexpr int QQ = decltype(q)::value;
      if (a.force) k_out<QQ, S, true><<<blocks_for(a.cnt, 128), 128, 0, st>>>(a);
      else k_out<QQ, S, false><<<blocks_for(a.cnt, 128), 128, 0, st>>>(a);
    });
  }
  static void set_state(int Q, const SetStateArgs& a, cudaStream_t st) {
    if (a.cnt <= 0) return;
    with_q(Q, [&](auto q) { k_set_state<decltype(q)::value, S><<<blocks_for(a.cnt, 128), 128, 0, st>>>(a); });
  }
  static void gather_ghosts(int Q, const GatherGhostArgs& a, cudaStream_t st) {
    if (a.cnt <= 0) return;
    with_q(Q, [&](auto q) { k_gather_ghosts<decltype(q)::value, S><<<blocks_for(a.cnt, 128), 128, 0, st>>>(a); });
  }
  static unsigned reduce(int Q, ReduceArgs& a, cudaStream_t st) {
    const unsigned g = assign_blocks(a, 1, [&](int k) {
      const ReduceLevel& l = a.lev[k];
      const int64_t n = std::max(l.end - l.begin, l.obs_n);
      return std::min<int64_t>(std::max<int64_t>((n + kRedBlock<S> - 1) / kRedBlock<S>, 1), kReduceBlocks);
    });
    with_q(Q, [&](auto q) { k_reduce<decltype(q)::value, S><<<g, kRedBlock<S>, 0, st>>>(a); });
    return g;
  }
};

template <class S>
const Ops* make_ops() {
  static const Ops ops = {&Launch<S>::sc_interior,    &Launch<S>::sc_rest,
                          &Launch<S>::outlet,         &Launch<S>::source_moments,
                          &Launch<S>::fill_gfc,       &Launch<S>::fill_gff,   &Launch<S>::fill_rest,
                          &Launch<S>::init,           &Launch<S>::init_place, &Launch<S>::out,
                          &Launch<S>::set_state,
                          &Launch<S>::gather_ghosts,
                          &Launch<S>::reduce,         sizeof(S),              sizeof(typename Sto<S>::R)};
  return &ops;
}

}  // namespace dev
}  // namespace lbm
