// Per-link and per-site device functions of the pure-gauge step, shared by
// the single-lattice kernels (gauge.cu) and the multi-chain kernels
// (batch.cu), so that a chain in a batch runs the same arithmetic.
#pragma once

#include <type_traits>

#include "df64.cuh"
#include "fg_common.cuh"
#include "fg_kernels.h"

namespace fg {

// Tuning knobs of the staple kernel: minimum resident blocks of 128 threads
// per SM (register cap) and whether the loop over the three staple
// directions is unrolled.
#ifndef FG_STAPLE_MIN_BLOCKS
#define FG_STAPLE_MIN_BLOCKS 4
#endif
#ifndef FG_FORCE_UNROLL_NU
#define FG_FORCE_UNROLL_NU 0
#endif

// Changes dp, dm of the half index lex/2 when coordinate nu of c moves by
// +1 and -1 (periodic); the parity flips.  Only that coordinate moves, so the change
// is (v>>1) - (c>>1) in x and (v - c) times the half stride of nu otherwise,
// and the changes of two steps in different directions add.
__device__ __forceinline__ void cb_half_steps(const Geom& g, const int c[4], int nu, int& dp, int& dm) {
  const int cn = sel4(c, nu);
  const int ln = nu == 0 ? g.L[0] : (nu == 1 ? g.L[1] : (nu == 2 ? g.L[2] : g.L[3]));
  const int vp = cn + 1 == ln ? 0 : cn + 1;
  const int vm = cn == 0 ? ln - 1 : cn - 1;
  if (nu == 0) {
    dp = (vp >> 1) - (cn >> 1);
    dm = (vm >> 1) - (cn >> 1);
  } else {
    const int hs = nu == 1 ? g.Lxh : (nu == 2 ? g.Lxh * g.L[1] : g.Lxh * g.L[1] * g.L[2]);
    dp = (vp - cn) * hs;
    dm = (vm - cn) * hs;
  }
}

// Product of two special unitary matrices (a link and a link, or exp(iA)
// and a link): the anchored products for double-float links.
template <typename R>
__device__ __forceinline__ M3<R> link_mul(const M3<R>& a, const M3<R>& b) {
  if constexpr (std::is_same<R, DF>::value) return su3_mul(a, b);
  else return mul(a, b);
}

// reunitarize of a product of two unitary matrices, rows 0 and 1.  The
// corrections are a few roundings: they are formed to first order, the three
// side by side, and in double-float added in FP32 (the general form took 6% of
// a double-float 12-real trajectory, this one 2%); where their squares would
// show, the general form takes over.  The norms are summed with all terms of a
// square: anchored double-float sums leave errors of one sign in them, 6e-15
// of |U|^2 after every drift.
template <typename R> __device__ __forceinline__ void project_product(M3<R>& u) {
  constexpr bool kDF = std::is_same<R, DF>::value;
  typedef typename std::conditional<kDF, float, R>::type C;   // a correction
  constexpr C most = kDF ? C(0x1p-25f) : (std::is_same<R, double>::value ? C(0x1p-27) : C(0x1p-13f));
  R n0 = R(-1), n1 = R(-1);   // |row0|^2 - 1, |row1|^2 - 1
  C c0, c1, pr, pi;           // and <row0, row1>, with the signs of the corrections
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    n0 = fma(u.e[0][k].im, u.e[0][k].im, fma(u.e[0][k].re, u.e[0][k].re, n0));
    n1 = fma(u.e[1][k].im, u.e[1][k].im, fma(u.e[1][k].re, u.e[1][k].re, n1));
  }
  if constexpr (kDF) {
    Anchored re, im;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const Cx<DF> a = u.e[0][k], b = u.e[1][k];
      re.add(a.re, b.re);
      re.add(a.im, b.im);
      im.add(a.re, b.im);
      im.sub(a.im, b.re);
    }
    c0 = -0.5f * n0.hi;
    c1 = -0.5f * n1.hi;
    pr = -re.value().hi;
    pi = -im.value().hi;
  } else {
    Cx<R> p = cx<R>(R(0), R(0));
#pragma unroll
    for (int k = 0; k < 3; ++k) cmac_cj(p, u.e[0][k], u.e[1][k]);
    c0 = R(-0.5) * n0;
    c1 = R(-0.5) * n1;
    pr = -p.re;
    pi = -p.im;
  }
  if (fabs(c0) + fabs(c1) + fabs(pr) + fabs(pi) < most) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Cx<R>& a = u.e[0][k];
      Cx<R>& b = u.e[1][k];
      if constexpr (kDF) {
        const float x = a.re.hi, y = a.im.hi;
        b.re = df_add_f(b.re, fmaf(c1, b.re.hi, fmaf(pr, x, -pi * y)));
        b.im = df_add_f(b.im, fmaf(c1, b.im.hi, fmaf(pr, y, pi * x)));
        a.re = df_add_f(a.re, c0 * x);
        a.im = df_add_f(a.im, c0 * y);
      } else {
        const Cx<R> t = a;
        b.re = fma(pr, t.re, fma(-pi, t.im, fma(c1, b.re, b.re)));
        b.im = fma(pr, t.im, fma(pi, t.re, fma(c1, b.im, b.im)));
        a = cx<R>(fma(c0, t.re, t.re), fma(c0, t.im, t.im));
      }
    }
  } else {
    reunitarize(u);
  }
}

// Stores exp(i c P) u (FP32: drift_pair's x and y in place of c and `half`),
// re-projected onto SU(3) if reunit is set (then rows 0
// and 1 of the product suffice) and always with 12-real links: their third row
// is rebuilt as (row0 x row1)^*, whose norm is off by the sum of the other
// two's, and the next product mixes that back into them, so that the defect of
// links that are only multiplied doubles every 20 trajectories (FP64 and
// double-float links were off by 1e-11 and 2e-9 after 200, by 3e-3 and 1
// after 800).
template <typename R, int NC>
__device__ __forceinline__ void drift_store(R p[8], R c, R half, const M3<R>& u, const Gauge<R, NC>& Uout, int mu,
                                            int s, int reunit) {
#pragma unroll
  for (int k = 0; k < 8; ++k) p[k] *= c;
  M3<R> e;
  if constexpr (std::is_same<R, float>::value) e = expi_herm(alg_to_mat(p, half));
  else e = expi_herm(alg_to_mat(p));
  if (reunit) {
    M3<R> un = mul_rows01(e, u);
    reunitarize(un);
    Uout.store(mu, s, un);
  } else {
    M3<R> un = link_mul(e, u);
    if constexpr (NC == 6) project_product(un);
    Uout.store(mu, s, un);
  }
}

// What MODE does with link (s, mu), f^a = Im Tr(lambda^a U A) given: the force
// is beta6 f + ffw FF (FP32 kicks: kick_pair's a, w and b in place of beta6, ffw
// and ckick).
template <typename R, int NC, int MODE>
__device__ __forceinline__ void force_apply(const Gauge<R, NC>& U, const Mom<R>& P, const Mom<R>& F, const Mom<R>& FF,
                                            const Gauge<R, NC>& Ubase, const Gauge<R, NC>& Uout, int s, int mu,
                                            R f[8], R beta6, R ckick, R cdrift, R half, R cdisp, int reunit, R ffw) {
#pragma unroll
  for (int k = 0; k < 8; ++k) f[k] = f[k] * beta6;
  if (FF.p != nullptr) {
    R ff[8];
    FF.load(mu, s, ff);
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] = fma(ffw, ff[k], f[k]);
  }
  if (MODE == FM_STORE) {
    F.store(mu, s, f);
  } else if (MODE == FM_KICK || MODE == FM_KICK_DRIFT) {
    R p[8];
    P.load(mu, s, p);
#pragma unroll
    for (int k = 0; k < 8; ++k) p[k] = fma(-ckick, f[k], p[k]);
    P.store(mu, s, p);
    if (MODE == FM_KICK_DRIFT) {
      drift_store(p, cdrift, half, Ubase.load(mu, s), Uout, mu, s, reunit);
    }
  } else {  // FM_DISPLACE
    // The displaced links only serve one force evaluation and are then
    // dropped, so they are not re-projected: FP32 exp(i A) U is off unitarity
    // by roundings of either sign (tr U^dag U short by 5e-11 on average).
    (void)reunit;
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] *= -cdisp;
    const M3<R> e = expi_herm(alg_to_mat(f));
    Uout.store(mu, s, link_mul(e, U.load(mu, s)));
  }
}

// ---------------------------------------------------------------------------
// The Wilson force by staples: one thread sums the six staples of its link.
// FP32 lattices take this form, and FP64 and double-float ones whose links are
// not unitary to their precision (kUnitaryWithin below): the staple sum is the
// derivative of the action for any link matrices.

// Sum of the six staples that close a plaquette with U_mu(x).  Neighbour
// indices are formed with selects, so mu and nu may be run-time values
// without the coordinate array going to local memory; one copy of the body
// keeps the kernel small enough for the instruction cache.
template <typename R, int NC>
__device__ __forceinline__ M3<R> staple_sum(const Gauge<R, NC>& U, const Geom& g, const int c[4], int s, int mu) {
  M3<R> a;
  zero(a);
  // neighbours as half-index steps from s: x + mu, x +- nu flip the parity,
  // x + mu - nu keeps it
  const int par = s >= g.Vh;
  const int other = s + (par ? -g.Vh : g.Vh);
  int dmu, dmu_m;
  cb_half_steps(g, c, mu, dmu, dmu_m);
  (void)dmu_m;
  const int s_pmu = other + dmu;
#if FG_FORCE_UNROLL_NU
#pragma unroll
#else
#pragma unroll 1
#endif
  for (int k = 1; k < 4; ++k) {
    const int nu = (mu + k) & 3;
    int dp, dm;
    cb_half_steps(g, c, nu, dp, dm);
    const int s_mnu = other + dm;
    if constexpr (std::is_same<R, DF>::value) {
      // Double-float: both staples of the plane as X Y^dag Z with run-time
      // daggers,
      //   upper  U_nu(x+mu)          U_mu(x+nu)^dag U_nu(x)^dag,
      //   lower  U_nu(x+mu-nu)^dag   U_mu(x-nu)^dag U_nu(x-nu),
      // their two products through one loop body (instruction cache), by the
      // anchored products of df64.cuh: links off unitarity by 1e-7, as
      // single precision leaves them, stay within the anchor's grid.
#pragma unroll 1
      for (int up = 1; up >= 0; --up) {
        M3<DF> l = dagger_if(U.load(nu, up ? s_pmu : s + dm + dmu), !up);
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
          const int sr = q ? (up ? s : s_mnu) : (up ? other + dp : s_mnu);
          l = su3_mul(l, dagger_if(U.load(q ? nu : mu, sr), q ? up != 0 : true));
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) a.e[i][j] = a.e[i][j] + l.e[i][j];
      }
    } else {
      {
        // upper: U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
        const M3<R> t = mul_nd(U.load(nu, s_pmu), U.load(mu, other + dp));
        mac_nd(a, t, U.load(nu, s));
      }
      {
        // lower: U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu) = (U_mu(x-nu) U_nu(x+mu-nu))^dag U_nu(x-nu)
        const M3<R> t = mul(U.load(mu, s_mnu), U.load(nu, s + dm + dmu));
        mac_dn(a, t, U.load(nu, s_mnu));
      }
    }
  }
  return a;
}

// f^a = Im Tr(lambda^a U A) for the staple sum a.
template <typename R> __device__ __forceinline__ void staple_force(const M3<R>& u, const M3<R>& a, R f[8]) {
  if constexpr (std::is_same<R, DF>::value) {
    // a / 8 (exact) has columns of norm 3/4 at most: within the anchored
    // products' bounds
    M3<DF> a8;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        a8.e[i][j] = cx<DF>(DF(a.e[i][j].re.hi * 0.125f, a.e[i][j].re.lo * 0.125f),
                            DF(a.e[i][j].im.hi * 0.125f, a.e[i][j].im.lo * 0.125f));
    im_tr_gellmann(su3_mul(u, a8), f);
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] = f[k] * 8.0f;
  } else {
    im_tr_gellmann(mul(u, a), f);
  }
}

template <typename R, int NC, int MODE>
__device__ __forceinline__ void force_link_staples(const Gauge<R, NC>& U, const Mom<R>& P, const Mom<R>& F,
                                                   const Mom<R>& FF, const Gauge<R, NC>& Ubase,
                                                   const Gauge<R, NC>& Uout, const Geom& g, const int c[4], int s,
                                                   int mu, R beta6, R ckick, R cdrift, R half, R cdisp, int reunit,
                                                   R ffw) {
  const M3<R> a = staple_sum(U, g, c, s, mu);
  R f[8];
  staple_force(U.load(mu, s), a, f);
  force_apply<R, NC, MODE>(U, P, F, FF, Ubase, Uout, s, mu, f, beta6, ckick, cdrift, half, cdisp, reunit, ffw);
}

// Whether the FP32 12-real force kernels share the upper-staple products of
// a plane between its two links through shared memory (below).  With 12-real
// links every load rebuilds a row, and the two loads a shared product saves
// pay for the barrier and the shared memory: 418 vs 437 us per launch at
// 32^4.  With 18-real links the same change executed 8% fewer instructions
// but ran 2% slower (426 vs 416 us; the slots take L1 capacity from the
// neighbour loads and the barrier stalls), and the FP64 kernels would need
// 55 KB of slots per block.
#ifndef FG_FORCE_SHARED_T
#define FG_FORCE_SHARED_T 1
#endif
// Resident blocks per SM of the sharing kernel (its register cap) and its
// preferred shared-memory carveout in percent of the SM's maximum (44%: the
// 100 KB configuration; five blocks of 32 sites: 1.5% faster than six).
#ifndef FG_FORCE_SHARED_MIN_BLOCKS
#define FG_FORCE_SHARED_MIN_BLOCKS 5
#endif
#ifndef FG_FORCE_CARVEOUT
#define FG_FORCE_CARVEOUT 44
#endif

// Upper staples of the plane (mu, nu) at x, for its two links: with
// T_{mu,nu} = U_nu(x+mu) U_mu(x+nu)^dag, the upper staple of U_mu(x) is
// T U_nu(x)^dag and that of U_nu(x) is U_mu(x+nu) U_nu(x+mu)^dag U_mu(x)^dag
// = T^dag U_mu(x)^dag = (U_mu(x) T)^dag.  The four direction threads of a
// site are in one block: thread mu computes T_{mu,mu+1} and, for mu < 2,
// T_{mu,mu+2} (6 products per site, 1 or 2 per thread), keeps its own term
// and leaves T in shared memory; after a barrier the other thread of each
// plane reads it.  A site's four links then take 46 3x3 products instead of
// 52 and two fewer link loads per shared plane.  Slots: T_{mu,mu+1} in mu,
// T_{mu,mu+2} in 4 + mu; entries as (re, im) pairs, site-minor.
// The block is NS sites (threadIdx.x) x 4 directions (threadIdx.y); tsh has
// room for the six slots of its NS sites.  Every thread of the block must
// call this (it holds a barrier); ok = false threads only take part in the
// barrier.  The caller separates two calls on the same tsh by a barrier.
template <typename R, int NC>
constexpr bool kForceSharedT = FG_FORCE_SHARED_T && std::is_same<R, float>::value && NC == 6;
template <int NC>
constexpr int kStapleMinBlocks = kForceSharedT<float, NC> ? FG_FORCE_SHARED_MIN_BLOCKS : FG_STAPLE_MIN_BLOCKS;

template <int NC, int MODE, int NS>
__device__ __forceinline__ void force_link_shared(float2 (*tsh)[9][NS], bool ok, int s, const Gauge<float, NC>& U,
                                                  const Mom<float>& P, const Mom<float>& F, const Mom<float>& FF,
                                                  const Gauge<float, NC>& Ubase, const Gauge<float, NC>& Uout,
                                                  const Geom& g, float beta6, float ckick, float cdrift,
                                                  float half, float cdisp, int reunit, float ffw) {
  const int x = threadIdx.x;
  const int mu = threadIdx.y;
  M3<float> a;
  zero(a);
  int c[4], par;
  if (ok) {
    cb_coords(g, s, c, par);
    const int other = s + (par ? -g.Vh : g.Vh);
    int dmu, dmu_m;
    cb_half_steps(g, c, mu, dmu, dmu_m);
    (void)dmu_m;
    const int s_pmu = other + dmu;
#pragma unroll 1
    for (int k = 1; k < 4; ++k) {
      const int nu = (mu + k) & 3;
      int dp, dm;
      cb_half_steps(g, c, nu, dp, dm);
      if (k == 1 || (k == 2 && mu < 2)) {
        const M3<float> t = mul_nd(U.load(nu, s_pmu), U.load(mu, other + dp));
        const int slot = k == 1 ? mu : 4 + mu;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) tsh[slot][3 * i + j][x] = make_float2(t.e[i][j].re, t.e[i][j].im);
        mac_nd(a, t, U.load(nu, s));
      }
      {
        // lower: (U_mu(x-nu) U_nu(x+mu-nu))^dag U_nu(x-nu)
        const int s_mnu = other + dm;
        const M3<float> t = mul(U.load(mu, s_mnu), U.load(nu, s + dm + dmu));
        mac_dn(a, t, U.load(nu, s_mnu));
      }
    }
  }
  __syncthreads();
  if (!ok) return;
  // planes whose T the other thread left: p = mu - 1 (slot p) and, for
  // mu >= 2, p = mu - 2 (slot 4 + p); add (U_p(x) T_{p,mu})^dag
#pragma unroll 1
  for (int r = 0; r < 2; ++r) {
    if (r == 1 && mu < 2) break;
    const int p = r == 0 ? ((mu + 3) & 3) : mu - 2;
    const int slot = r == 0 ? p : 4 + p;
    M3<float> t;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const float2 v = tsh[slot][3 * i + j][x];
        t.e[i][j] = cx<float>(v.x, v.y);
      }
    const M3<float> up = U.load(p, s);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        // a_ij += conj((U_p T)_ji)
        Cx<float> acc = conj(a.e[i][j]);
        cmac(acc, up.e[j][0], t.e[0][i]);
        cmac(acc, up.e[j][1], t.e[1][i]);
        cmac(acc, up.e[j][2], t.e[2][i]);
        a.e[i][j] = conj(acc);
      }
  }
  float f[8];
  staple_force(U.load(mu, s), a, f);
  force_apply<float, NC, MODE>(U, P, F, FF, Ubase, Uout, s, mu, f, beta6, ckick, cdrift, half, cdisp, reunit, ffw);
}

// ---------------------------------------------------------------------------
// The Wilson force by plaquettes (double-float and FP64 links).
//
// The four links of a plaquette share its force.  With
//   W_{mu nu}(x) = U_mu(x) U_nu(x+mu) (U_nu(x) U_mu(x+nu))^dag,   mu < nu,
// and Q the Hermitian traceless part of W (W = ... + i Q),
//   * U_mu(x) takes +Q and U_nu(x) takes -Q (their products with the staple
//     are W and W^dag);
//   * U_mu(x+nu) takes -U_nu(x)^dag Q U_nu(x) and U_nu(x+mu) takes
//     +U_mu(x)^dag Q U_mu(x) (the same closed path read from another corner;
//     this step uses U^dag U = 1: lattices whose links are not unitary to
//     their precision take the staple sums, see kUnitaryWithin).
// plaquette_kernel forms Q once for every site and plane (two products and
// half of a third), link_force_kernel sums six of them for every link, three
// of them rotated by one neighbour link (90 + 48 multiply-adds, H being
// Hermitian).  A site then takes 6 x 306 + 12 x 138 = 3492 multiply-adds
// instead of the 4 x 13 x 108 = 5616 of a staple sum for every link.
// Double-float and FP64 forces are bound by that arithmetic (FP32 and FP64
// issue), so they take this form: an FG trajectory against the staple sums over
// the same rows takes 1.65 instead of 2.25 ms (double-float 16^4), 7.56 instead
// of 10.3 (24^4), 7.92 instead of 10.1 (FP64 16^4), and on small lattices 0.37
// instead of 0.39 ms (double-float 8^4) and 0.67 instead of 0.85 (FP64 4^4).
// The FP32 force executes 18% fewer instructions
// this way but waits for the memory traffic of Q (193 + 233 us a launch pair
// against 405 us at 32^4; 12% slower at 8^4): it stays with the staples.  One
// launch of both kinds of work, link blocks waiting for the plaquettes they
// read, was 5 to 25% slower than two launches (idle SMs, spilled registers).
// Q is kept in the momenta's layout, [plane][2][site], by its entries
// (q00, q11, Re q01, Im q01, Re q02, Im q02, Re q12, Im q12).

// Most threads of a block of the two kernels, and resident blocks of that
// size asked of the register allocator: 168 and 128 registers a thread, where
// neither spills (plaquettes at 128 registers: 5-7% slower in double-float).
#ifndef FG_PLAQ_THREADS
#define FG_PLAQ_THREADS 128
#endif
#ifndef FG_PLAQ_MIN_BLOCKS
#define FG_PLAQ_MIN_BLOCKS 3
#endif
#ifndef FG_LINK_MIN_BLOCKS
#define FG_LINK_MIN_BLOCKS 4
#endif
constexpr int kForceThreads = FG_PLAQ_THREADS;

// One lattice of a launch: its geometry, coupling and the byte offsets of its
// links, momenta and plaquette field in the launch's buffers.
struct ChainDesc {
  Geom g;
  long long goff, moff, woff;
  long long soff;  // offset of its sites in per-site arrays
  double beta, beta6;          // beta, beta / 6
  float beta6_hi, beta6_lo;    // beta / 6 as a double-float: no FP64 arithmetic (1/64 of the FP32 rate) there
  int tile0, ntiles;           // its tiles (batch.cu)
};
template <typename R> __device__ __forceinline__ R beta6_of(const ChainDesc& cd);
template <> __device__ __forceinline__ double beta6_of<double>(const ChainDesc& cd) { return cd.beta6; }
template <> __device__ __forceinline__ float beta6_of<float>(const ChainDesc& cd) { return cd.beta6_hi; }
template <> __device__ __forceinline__ DF beta6_of<DF>(const ChainDesc& cd) { return DF(cd.beta6_hi, cd.beta6_lo); }

// Largest entry of U U^dag - 1 with which a lattice takes the plaquette form.
// A force by plaquettes is off by about the defect of its links (the staple
// sums by none of it), and one FG trajectory's dH by some 20 times the
// defect's mean size on 6^4, growing with the root of the volume: below the
// lines, less than the rounding of the forces and sums puts into dH (FP64
// 1e-12, double-float 1e-10 there).  Links held in single precision lie at
// 1e-7, links made unitary in 64 bits at 1e-15, and a chain that is never
// re-projected moves away from there with the root of its length: FP64 18-real
// chains reach 7e-14 and double-float ones 1.8e-11 in 800 trajectories of 16
// drifts.  The defect is therefore taken anew after every trajectory.
template <typename R>
constexpr double kUnitaryWithin = std::is_same<R, double>::value ? 0x1p-42 : 0x1p-35;

// Whether an entry of U U^dag - 1 is larger than `most` (or not a number).
// In double-float by anchored sums (df64.cuh; those of the diagonal start at
// -1): general double-float FMAs took 38 us over a 16^4 lattice.
template <typename R> __device__ __forceinline__ bool off_unitary(const M3<R>& u, R most) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j <= i; ++j) {
      R re = R(i == j ? -1 : 0), im = R(0);
      if constexpr (std::is_same<R, DF>::value) {
        Anchored x, y;
        if (i == j) x.t = 2.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          x.add(u.e[i][k].re, u.e[j][k].re);
          x.add(u.e[i][k].im, u.e[j][k].im);
          if (i != j) {
            y.add(u.e[i][k].im, u.e[j][k].re);
            y.sub(u.e[i][k].re, u.e[j][k].im);
          }
        }
        re = x.value();
        im = y.value();
      } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          re = fma(u.e[i][k].re, u.e[j][k].re, fma(u.e[i][k].im, u.e[j][k].im, re));
          if (i != j) im = fma(u.e[i][k].im, u.e[j][k].re, fma(-u.e[i][k].re, u.e[j][k].im, im));
        }
      }
      ok = ok && fabs(re) < most && fabs(im) < most;
    }
  return !ok;
}

// Plane pl = 0..5 as directions mu < nu, and back.
__device__ __forceinline__ void plane_dirs(int pl, int& mu, int& nu) {
  mu = pl < 3 ? 0 : (pl < 5 ? 1 : 2);
  nu = pl < 3 ? pl + 1 : (pl < 5 ? pl - 1 : 3);
}
__device__ __forceinline__ int plane_of(int a, int b) {
  const int mu = a < b ? a : b, nu = a < b ? b : a;
  return mu == 0 ? nu - 1 : (mu == 1 ? nu + 1 : 5);
}

// q = Hermitian traceless part of W_pl(s).
template <typename R, int NC>
__device__ __forceinline__ void plaquette_herm(const Gauge<R, NC>& U, const Geom& g, int s, int pl, R q[8]) {
  int c[4], par, mu, nu;
  cb_coords(g, s, c, par);
  plane_dirs(pl, mu, nu);
  const int other = s + (par ? -g.Vh : g.Vh);
  int dmu, dnu, dm;
  cb_half_steps(g, c, mu, dmu, dm);
  cb_half_steps(g, c, nu, dnu, dm);
  (void)dm;
  if constexpr (std::is_same<R, DF>::value) {
    // both corner products through one loop body (instruction cache)
    M3<DF> a, b;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      const M3<DF> m = su3_mul(U.load(k ? nu : mu, s), U.load(k ? mu : nu, other + (k ? dnu : dmu)));
      if (k) b = m;
      else a = m;
    }
    // half of a (exact) keeps the sums of two entries of W within the
    // anchored accumulator's [-1, 1]
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        a.e[i][j] = cx<DF>(DF(0.5f * a.e[i][j].re.hi, 0.5f * a.e[i][j].re.lo),
                           DF(0.5f * a.e[i][j].im.hi, 0.5f * a.e[i][j].im.lo));
    DF d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Anchored t;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        t.add(a.e[i][k].im, b.e[i][k].re);
        t.sub(a.e[i][k].re, b.e[i][k].im);
      }
      d[i] = t.value();
    }
    constexpr DF third(1.0 / 3.0);
    const DF tr = (d[0] + d[1] + d[2]) * third;
    q[0] = (d[0] - tr) * 2.0f;
    q[1] = (d[1] - tr) * 2.0f;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const int i = p < 2 ? 0 : 1, j = p == 0 ? 1 : 2;
      Anchored re, im;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        re.add(a.e[i][k].im, b.e[j][k].re);
        re.sub(a.e[i][k].re, b.e[j][k].im);
        re.add(a.e[j][k].im, b.e[i][k].re);
        re.sub(a.e[j][k].re, b.e[i][k].im);
        im.sub(a.e[i][k].re, b.e[j][k].re);
        im.sub(a.e[i][k].im, b.e[j][k].im);
        im.add(a.e[j][k].re, b.e[i][k].re);
        im.add(a.e[j][k].im, b.e[i][k].im);
      }
      q[2 + 2 * p] = re.value();
      q[3 + 2 * p] = im.value();
    }
  } else {
    const M3<R> a = mul(U.load(mu, s), U.load(nu, other + dmu));
    const M3<R> b = mul(U.load(nu, s), U.load(mu, other + dnu));
    R d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      R t = R(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        t = fma(a.e[i][k].im, b.e[i][k].re, t);
        t = fma(-a.e[i][k].re, b.e[i][k].im, t);
      }
      d[i] = t;
    }
    const R tr = (d[0] + d[1] + d[2]) * R(1.0 / 3.0);
    q[0] = d[0] - tr;
    q[1] = d[1] - tr;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const int i = p < 2 ? 0 : 1, j = p == 0 ? 1 : 2;
      R re = R(0), im = R(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        re = fma(a.e[i][k].im, b.e[j][k].re, re);
        re = fma(-a.e[i][k].re, b.e[j][k].im, re);
        re = fma(a.e[j][k].im, b.e[i][k].re, re);
        re = fma(-a.e[j][k].re, b.e[i][k].im, re);
        im = fma(-a.e[i][k].re, b.e[j][k].re, im);
        im = fma(-a.e[i][k].im, b.e[j][k].im, im);
        im = fma(a.e[j][k].re, b.e[i][k].re, im);
        im = fma(a.e[j][k].im, b.e[i][k].im, im);
      }
      q[2 + 2 * p] = R(0.5) * re;
      q[3 + 2 * p] = R(0.5) * im;
    }
  }
}

// acc += u^dag H u for the Hermitian traceless H given by h (entries as
// above), a column of H u at a time.
template <typename R>
__device__ __forceinline__ void rotate_add(R acc[8], const R h[8], const M3<R>& u) {
  const R h22 = -(h[0] + h[1]);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const Cx<R> u0 = u.e[0][j], u1 = u.e[1][j], u2 = u.e[2][j];
    Cx<R> v[3];
    v[0] = cx<R>(h[0] * u0.re, h[0] * u0.im);
    cmac(v[0], cx<R>(h[2], h[3]), u1);
    cmac(v[0], cx<R>(h[4], h[5]), u2);
    v[1] = cx<R>(h[1] * u1.re, h[1] * u1.im);
    cmac_cj(v[1], cx<R>(h[2], h[3]), u0);
    cmac(v[1], cx<R>(h[6], h[7]), u2);
    v[2] = cx<R>(h22 * u2.re, h22 * u2.im);
    cmac_cj(v[2], cx<R>(h[4], h[5]), u0);
    cmac_cj(v[2], cx<R>(h[6], h[7]), u1);
    if (j < 2) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        acc[j] = fma(u.e[k][j].re, v[k].re, acc[j]);
        acc[j] = fma(u.e[k][j].im, v[k].im, acc[j]);
      }
    }
#pragma unroll
    for (int i = 0; i < j; ++i) {
      const int p = i + j;  // (0,1) -> 1, (0,2) -> 2, (1,2) -> 3
      Cx<R> t = cx<R>(acc[2 * p], acc[2 * p + 1]);
#pragma unroll
      for (int k = 0; k < 3; ++k) cmac_cj(t, u.e[k][i], v[k]);
      acc[2 * p] = t.re;
      acc[2 * p + 1] = t.im;
    }
  }
}

// Double-float: the entries of H u and u^dag H u and their partial sums are
// bounded by the norm of H, which stays below the anchored products' 1 unless
// the plaquette is far from the unit matrix (Q's eigenvalues are sines less
// their mean, 4/3 at most); beyond, the accumulator's grid is twice as coarse.
// (H / 2 is always within the bound but doubles the rounding of every force.)
template <>
__device__ __forceinline__ void rotate_add<DF>(DF acc[8], const DF h[8], const M3<DF>& u) {
  const DF h22 = -(h[0] + h[1]);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    Cx<DF> v[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      Anchored re, im;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const Cx<DF> x = u.e[k][j];
        if (k == r) {
          const DF d = r == 0 ? h[0] : (r == 1 ? h[1] : h22);
          re.add(d, x.re);
          im.add(d, x.im);
        } else {
          const int p = k + r;  // the entry above the diagonal; its conjugate below
          const DF hr = h[2 * p], hi = h[2 * p + 1];
          re.add(hr, x.re);
          im.add(hr, x.im);
          if (k > r) {
            re.sub(hi, x.im);
            im.add(hi, x.re);
          } else {
            re.add(hi, x.im);
            im.sub(hi, x.re);
          }
        }
      }
      v[r] = cx<DF>(re.value(), im.value());
    }
#pragma unroll
    for (int i = 0; i <= j; ++i) {
      if (i == 2) continue;  // the trace is zero
      Anchored re, im;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        re.add(u.e[k][i].re, v[k].re);
        re.add(u.e[k][i].im, v[k].im);
        if (i < j) {
          im.add(u.e[k][i].re, v[k].im);
          im.sub(u.e[k][i].im, v[k].re);
        }
      }
      if (i == j) {
        acc[i] = acc[i] + re.value();
      } else {
        acc[2 * (i + j)] = acc[2 * (i + j)] + re.value();
        acc[2 * (i + j) + 1] = acc[2 * (i + j) + 1] + im.value();
      }
    }
  }
}

template <typename R> __device__ __forceinline__ R flip_if(R x, bool n) { return n ? -x : x; }

// f^a = Im Tr(lambda^a U_mu(s) A_mu(s)), A the staple sum, from the
// plaquette field W of these links.
template <typename R, int NC>
__device__ __forceinline__ void link_force(const Gauge<R, NC>& U, const Mom<R>& W, const Geom& g, int s, int mu,
                                           R f[8]) {
  int c[4], par;
  cb_coords(g, s, c, par);
  const int other = s + (par ? -g.Vh : g.Vh);
  R acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = R(0);
  // one copy of the body (instruction cache)
#pragma unroll 1
  for (int d = 1; d < 4; ++d) {
    const int nu = (mu + d) & 3;
    const int pl = plane_of(mu, nu);
    int dp, dm;
    cb_half_steps(g, c, nu, dp, dm);
    (void)dp;
    const int sm = other + dm;  // x - nu
    R h[8];
    W.load(pl, s, h);
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = acc[k] + flip_if(h[k], mu > nu);
    W.load(pl, sm, h);
#pragma unroll
    for (int k = 0; k < 8; ++k) h[k] = flip_if(h[k], mu < nu);
    rotate_add(acc, h, U.load(nu, sm));
  }
  const R two = R(2.0f), s3 = R(1.73205080756887729353);
  f[0] = two * acc[2];
  f[1] = -(two * acc[3]);
  f[2] = acc[0] - acc[1];
  f[3] = two * acc[4];
  f[4] = -(two * acc[5]);
  f[5] = two * acc[6];
  f[6] = -(two * acc[7]);
  f[7] = s3 * (acc[0] + acc[1]);
}

template <typename R, int NC, int MODE>
__device__ __forceinline__ void force_link_plaquettes(const Gauge<R, NC>& U, const Mom<R>& W, const Mom<R>& P,
                                                      const Mom<R>& F, const Mom<R>& FF, const Gauge<R, NC>& Ubase,
                                                      const Gauge<R, NC>& Uout, const Geom& g, int s, int mu, R beta6,
                                                      R ckick, R cdrift, R half, R cdisp, int reunit,
                                                      R ffw) {
  R f[8];
  link_force(U, W, g, s, mu, f);
  force_apply<R, NC, MODE>(U, P, F, FF, Ubase, Uout, s, mu, f, beta6, ckick, cdrift, half, cdisp, reunit, ffw);
}

// U_out(s, mu) = exp(i c P) U_in(s, mu), the exact T-hat flow of section 2.
template <typename R, int NC>
__device__ __forceinline__ void drift_link(const Gauge<R, NC>& Uin, const Mom<R>& P, const Gauge<R, NC>& Uout,
                                           int s, int mu, R c, R half, int reunit) {
  R p[8];
  P.load(mu, s, p);
  drift_store(p, c, half, Uin.load(mu, s), Uout, mu, s, reunit);
}

// Per-site energy h(x) = T(x) + S_G(x) (T = 0 if P is null), with
// S_G(x) = sum_{mu<nu} beta (1 - Re Tr P_mu,nu(x) / 3) = beta6 - beta3 sum Re Tr
// (beta6 = 6 beta, beta3 = beta / 3): v[0] = S_G(x), v[1] = T(x); mode 0
// stores h0[s] = h(x), mode 1 sets v[2] = h(x) - h0[s].  If sg_in is given,
// S_G(x) is read from it instead of recomputed (the links have not changed
// since it was stored); if sg_out is given, S_G(x) is stored.  A is the type
// of the per-site values: double, or DF for FP32 and double-float fields,
// which keeps FP64 arithmetic (1/64 of the FP32 rate on GB300) out of the
// kernel.  Sums of FP32 terms are double-float in either case (each p^2
// split exactly by an FMA, each plaquette trace added with two_sum);
// double-float fields compute and sum in double-float, FP64 fields in FP64.
template <typename A> __device__ __forceinline__ A acc_of(DF x);
template <> __device__ __forceinline__ DF acc_of<DF>(DF x) { return x; }
template <> __device__ __forceinline__ double acc_of<double>(DF x) { return double(x); }

template <typename R, int NC, typename A>
__device__ __forceinline__ void site_energy(const Gauge<R, NC>& U, const Mom<R>& P, const Geom& g, int s,
                                            A beta6, A beta3, int mode, A* __restrict__ h0, A v[3],
                                            const A* __restrict__ sg_in = nullptr, A* __restrict__ sg_out = nullptr) {
  constexpr bool kDF = std::is_same<R, float>::value;
  constexpr bool kDD = std::is_same<R, DF>::value;
  static_assert(kDF || kDD || std::is_same<A, double>::value, "FP64 fields keep FP64 per-site values");
  A t = A(0);
  if (P.p != nullptr) {
    DF tdf(0.0f);
    double t64 = 0.0;
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      R p[8];
      P.load(mu, s, p);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if constexpr (kDF) {
          const float sq = __fmul_rn(p[k], p[k]);
          tdf = tdf + DF(sq, __fmaf_rn(p[k], p[k], -sq));
        } else if constexpr (kDD) {
          tdf = fma(p[k], p[k], tdf);
        } else {
          t64 += double(p[k]) * double(p[k]);
        }
      }
    }
    if constexpr (kDF || kDD) t = acc_of<A>(tdf) * A(0.5f);
    else t = A(0.5 * t64);
  }
  A sg;
  if (sg_in != nullptr) {
    sg = sg_in[s];
  } else {
    int c[4], par;
    cb_coords(g, s, c, par);
    // x + mu as a half-index step from s (cb_half_steps)
    const int other = s + (par ? -g.Vh : g.Vh);
    int dp[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      int dm;
      cb_half_steps(g, c, mu, dp[mu], dm);
      (void)dm;
    }
    DF trdf(0.0f);
    double tr64 = 0.0;
    if constexpr (kDD) {
      // double-float links: the plaquette's two products by the anchored
      // products, one copy of the code for the six planes (x, y, z, t as
      // mu, nu with mu < nu; the planes' half-index steps by selects)
#pragma unroll 1
      for (int pl = 0; pl < 6; ++pl) {
        const int mu = pl < 3 ? 0 : (pl < 5 ? 1 : 2);
        const int nu = pl < 3 ? pl + 1 : (pl < 5 ? pl - 1 : 3);
        const int dmu = sel4(dp, mu), dnu = sel4(dp, nu);
        M3<DF> pr[2];
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
          // U_mu(x) U_nu(x+mu), then U_nu(x) U_mu(x+nu)
          const M3<DF> l = U.load(q ? nu : mu, s);
          const M3<DF> r = U.load(q ? mu : nu, other + (q ? dnu : dmu));
          const M3<DF> m = su3_mul(l, r);
          if (q) pr[1] = m;
          else pr[0] = m;
        }
        trdf = trdf + re_tr_mul_nd(pr[0], pr[1]);
      }
    } else {
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        const M3<R> umu = U.load(mu, s);
#pragma unroll
        for (int nu = mu + 1; nu < 4; ++nu) {
          const M3<R> a = mul(umu, U.load(nu, other + dp[mu]));
          const M3<R> b = mul(U.load(nu, s), U.load(mu, other + dp[nu]));
          if constexpr (kDF) trdf = trdf + DF(float(re_tr_mul_nd(a, b)));
          else tr64 += double(re_tr_mul_nd(a, b));
        }
      }
    }
    if constexpr (kDF || kDD) sg = beta6 - beta3 * acc_of<A>(trdf);
    else sg = beta6 - beta3 * A(tr64);
  }
  if (sg_out != nullptr) sg_out[s] = sg;
  v[0] = sg;
  v[1] = t;
  const A h = sg + t;
  if (mode == 0) h0[s] = h;
  else if (mode == 1) v[2] = h - h0[s];
}

// Box-Muller on two 32-bit uniforms, u1 in (0, 1], u2 in [0, 1), evaluated
// in the precision of the momenta (GB300's FP64 unit is slow, and FP32
// momenta cannot hold more than an FP32 draw).
template <typename R>
__device__ __forceinline__ void box_muller(uint32_t a, uint32_t b, R& z0, R& z1) {
  const R u1 = (R(a) + R(1)) * R(2.3283064365386963e-10);
  const R u2 = R(b) * R(2.3283064365386963e-10);
  const R r = sqrt(R(-2) * log(u1));
  R sn, cs;
  sincospi(R(2) * u2, &sn, &cs);
  z0 = r * cs;
  z1 = r * sn;
}

// Double-float fields take FP32 draws: the Gaussian deviates need no more
// than FP32 resolution, and every later use of them (kinetic term, MD) is
// exact to double-float rounding for whatever value was drawn.
template <>
__device__ __forceinline__ void box_muller<DF>(uint32_t a, uint32_t b, DF& z0, DF& z1) {
  float x0, x1;
  box_muller<float>(a, b, x0, x1);
  z0 = DF(x0);
  z1 = DF(x1);
}

// Unit-Gaussian momenta of link (s, mu): two Philox-4x32-10 draws with
// counter (4 lex + mu, draw, stream, half); stream 0 = one lattice,
// stream 3 + chain for the chains of a batch.
template <typename R>
__device__ __forceinline__ void refresh_link(const Mom<R>& P, const Geom& g, int s, int mu, uint32_t k0, uint32_t k1,
                                             uint32_t draw, uint32_t stream) {
  int c[4], par;
  cb_coords(g, s, c, par);
  const uint32_t lex = (uint32_t)(c[0] + g.L[0] * (c[1] + g.L[1] * (c[2] + g.L[2] * c[3])));
  R p[8];
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    uint32_t ctr[4] = {lex * 4u + (uint32_t)mu, draw, stream, (uint32_t)half};
    Philox::rounds(ctr, k0, k1);
    box_muller<R>(ctr[0], ctr[1], p[4 * half + 0], p[4 * half + 1]);
    box_muller<R>(ctr[2], ctr[3], p[4 * half + 2], p[4 * half + 3]);
  }
  P.store(mu, s, p);
}

}  // namespace fg
