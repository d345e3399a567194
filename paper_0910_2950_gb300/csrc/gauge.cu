// Pure-gauge kernels of the force-gradient HMC step (sm_103a).
//
//  * staple_force_kernel (FP32), plaquette_kernel and link_force_kernel
//    (double-float and FP64; staple_rows_kernel where unitarity_kernel finds
//    the links off unitarity): Wilson force F^a = (beta/6) Im Tr(lambda^a U A), A the sum of the
//    link's staples (the S-hat vector field of section 3), fused with what
//    the integrator does next on the same link: store it, kick the momentum,
//    kick then drift the link, or displace the link along the force for the
//    force-gradient step of Table 1 (U' = exp(-i dt^2/24 F) U).
//  * drift_kernel: the exact T-hat flow U <- exp(i c P) U (section 2).
//  * energy_kernel: per-site T(x) + S_G(x), in double-float for FP32 fields
//    and FP64 for FP64 fields, block partial sums for the dH of section 5
//    (summed as site-by-site differences).
//  * refresh_momenta_kernel: unit-Gaussian momenta from a counter-based RNG.
//
// One thread per link (or plaquette); blocks take 32 consecutive half-sites of
// a parity in all directions, or some of their warps, so the links of a site
// and their staples share L1/L2 lines.
#include <type_traits>

#include "fg_common.cuh"
#include "fg_kernels.h"
#include "gauge_device.cuh"

namespace fg {

static Geom to_dev(const GeomH& h) {
  Geom g;
  for (int i = 0; i < 4; ++i) g.L[i] = h.L[i];
  g.Lxh = h.Lxh; g.Vh = h.Vh; g.V = h.V;
  g.dLxh = make_fastdiv((uint32_t)h.Lxh);
  g.dLy = make_fastdiv((uint32_t)h.L[1]);
  g.dLz = make_fastdiv((uint32_t)h.L[2]);
  return g;
}

constexpr int kSitesPerBlock = 64;
constexpr int kSms = 152;  // SMs of a GB300

// Warps of a block: `most` while that leaves two blocks for every SM, fewer on
// small lattices, so that their few warps spread over the SMs instead of
// queueing on some of them.
static inline int warps_per_block(long long warps, int most) {
  int w = most;
  while (w > 1 && warps < (long long)w * 2 * kSms) w /= 2;
  return w;
}


// One thread a link: a block takes 32 half-sites of one parity in all four
// directions, blocks of the two parities side by side.  (Both parities in one
// block of 256 threads: 18% slower at 8^4, 1% at 24^4 and 32^4.)
constexpr int kStapleSites = 32;
template <int NC, int MODE>
__global__ void __launch_bounds__(4 * kStapleSites, kStapleMinBlocks<NC>)
    staple_force_kernel(Gauge<float, NC> U, Mom<float> P, Mom<float> F, Mom<float> FF, Gauge<float, NC> Ubase,
                        Gauge<float, NC> Uout, Geom g, float beta6, float ckick, float cdrift, float half, float cdisp,
                        int reunit, float ffw) {
  const int i = (int)(blockIdx.x >> 1) * kStapleSites + (int)threadIdx.x, s = (int)(blockIdx.x & 1) * g.Vh + i;
  const bool ok = i < g.Vh;
  if constexpr (kForceSharedT<float, NC>) {
    __shared__ float2 tsh[6][9][kStapleSites];
    force_link_shared<NC, MODE, kStapleSites>(tsh, ok, s, U, P, F, FF, Ubase, Uout, g, beta6, ckick, cdrift, half, cdisp, reunit,
                                    ffw);
  } else {
    if (!ok) return;
    int c[4], par;
    cb_coords(g, s, c, par);
    force_link_staples<float, NC, MODE>(U, P, F, FF, Ubase, Uout, g, c, s, (int)threadIdx.y, beta6, ckick, cdrift, half, cdisp,
                                 reunit, ffw);
  }
}

// The double-float and FP64 launches walk their lattices by warps (rows of 32
// consecutive half-sites of one parity): warp w takes part w % parts (a plane
// or a direction) of row w / parts; all parts and both parities of the same
// half-sites are in consecutive warps and share the links in L1.
struct RowSite {
  const ChainDesc* cd;
  int s, part;
};
__device__ __forceinline__ bool row_site(const ForceRows& r, int parts, RowSite& o) {
  const unsigned w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const unsigned q = w / (unsigned)parts;
  o.part = (int)(w - q * (unsigned)parts);
  const int row = (int)(q >> 1);
  if (row >= r.nrows) return false;
  const ChainDesc* cd = (const ChainDesc*)r.chains;
  int i = row * 32;
  if (r.rows != nullptr) {
    const int2 at = r.rows[row];
    cd += at.x;
    i = at.y;
  }
  i += (int)(threadIdx.x & 31);
  if (i >= cd->g.Vh) return false;
  o.cd = cd;
  o.s = (int)(q & 1) * cd->g.Vh + i;
  return true;
}

// Q of every site and plane (gauge_device.cuh).
template <typename R, int NC>
__global__ void __launch_bounds__(kForceThreads, FG_PLAQ_MIN_BLOCKS)
    plaquette_kernel(const __grid_constant__ ForceRows r, char* U, char* W) {
  RowSite o;
  if (!row_site(r, 6, o)) return;
  const Geom g = o.cd->g;
  Gauge<R, NC> u;
  u.p = U + o.cd->goff; u.V = g.V;
  Mom<R> w;
  w.p = W + o.cd->woff; w.V = g.V;
  R q[8];
  plaquette_herm(u, g, o.s, o.part, q);
  w.store(o.part, o.s, q);
}

// The force of every link from Q, and what MODE does with it.
template <typename R, int NC, int MODE>
__global__ void __launch_bounds__(kForceThreads, FG_LINK_MIN_BLOCKS)
    link_force_kernel(const __grid_constant__ ForceRows r, char* U, char* W, char* P, char* F, char* FF, char* Ubase,
                      char* Uout, R ckick, R cdrift, R half, R cdisp, int reunit, R ffw) {
  RowSite o;
  if (!row_site(r, 4, o)) return;
  const ChainDesc& cd = *o.cd;
  const Geom g = cd.g;
  Gauge<R, NC> u, ub, uo;
  u.p = U + cd.goff; u.V = g.V;
  ub.p = Ubase + cd.goff; ub.V = g.V;
  uo.p = Uout + cd.goff; uo.V = g.V;
  Mom<R> w, p, f, ff;
  w.p = W + cd.woff; w.V = g.V;
  p.p = P + cd.moff; p.V = g.V;
  f.p = F + cd.moff; f.V = g.V;
  ff.p = FF == nullptr ? nullptr : FF + cd.moff; ff.V = g.V;
  force_link_plaquettes<R, NC, MODE>(u, w, p, f, ff, ub, uo, g, o.s, o.part, beta6_of<R>(cd), ckick, cdrift, half, cdisp,
                                     reunit, ffw);
}

// The same from the staple sums (links that are not unitary to R).
template <typename R, int NC, int MODE>
__global__ void __launch_bounds__(kForceThreads, FG_LINK_MIN_BLOCKS)
    staple_rows_kernel(const __grid_constant__ ForceRows r, char* U, char* P, char* F, char* FF, char* Ubase,
                       char* Uout, R ckick, R cdrift, R half, R cdisp, int reunit, R ffw) {
  RowSite o;
  if (!row_site(r, 4, o)) return;
  const ChainDesc& cd = *o.cd;
  const Geom g = cd.g;
  Gauge<R, NC> u, ub, uo;
  u.p = U + cd.goff; u.V = g.V;
  ub.p = Ubase + cd.goff; ub.V = g.V;
  uo.p = Uout + cd.goff; uo.V = g.V;
  Mom<R> p, f, ff;
  p.p = P + cd.moff; p.V = g.V;
  f.p = F + cd.moff; f.V = g.V;
  ff.p = FF == nullptr ? nullptr : FF + cd.moff; ff.V = g.V;
  int c[4], par;
  cb_coords(g, o.s, c, par);
  force_link_staples<R, NC, MODE>(u, p, f, ff, ub, uo, g, c, o.s, o.part, beta6_of<R>(cd), ckick, cdrift, half, cdisp, reunit,
                                  ffw);
}

// flag[stride * lattice] = 1 where a link of the lattice is off unitarity by
// more than `most`.
template <typename R, int NC>
__global__ void __launch_bounds__(kForceThreads)
    unitarity_kernel(const __grid_constant__ ForceRows r, char* U, R most, double* __restrict__ flag, int stride) {
  RowSite o;
  const bool in = row_site(r, 4, o);
  bool off = false;
  if (in) {
    Gauge<R, NC> u;
    u.p = U + o.cd->goff; u.V = o.cd->g.V;
    off = off_unitary(u.load(o.part, o.s), most);
  }
  // lane 0 of a row is always one of its sites; one writer a warp
  if (__any_sync(0xffffffffu, off) && (threadIdx.x & 31) == 0)
    atomicExch((unsigned long long*)(flag + stride * (o.cd - (const ChainDesc*)r.chains)), 0x3ff0000000000000ull);  // 1.0
}

// One thread a link: warp w takes direction w mod 4 of 32 consecutive sites.
template <typename R, int NC>
__global__ void __launch_bounds__(256) drift_kernel(Gauge<R, NC> Uin, Mom<R> P, Gauge<R, NC> Uout,
                                                    int V, R c, R half, int reunit) {
  const unsigned w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int s = (int)(w >> 2) * 32 + (int)(threadIdx.x & 31);
  if (s >= V) return;
  drift_link(Uin, P, Uout, s, (int)(w & 3), c, half, reunit);
}

template <typename R, int NC>
__global__ void __launch_bounds__(256) unit_links_kernel(Gauge<R, NC> U, int V) {
  const int s = blockIdx.x * kSitesPerBlock + threadIdx.x;
  const int mu = threadIdx.y;
  if (s >= V) return;
  M3<R> u;
  identity(u);
  U.store(mu, s, u);
}

// Haar-random SU(3) link from 12 Gaussians (Philox counter (4 lex + mu, draw,
// stream 5, word)): Gram-Schmidt of two complex Gaussian rows gives the first
// two rows of a Haar U(3) matrix, which fix the SU(3) matrix with the third
// row (row1 x row2)^*; SU(3) is in one-to-one correspondence with such row
// pairs, so the result is Haar on SU(3).
template <typename R, int NC>
__global__ void __launch_bounds__(256) random_links_kernel(Gauge<R, NC> U, Geom g, uint32_t k0, uint32_t k1,
                                                           uint32_t draw) {
  const int s = blockIdx.x * kSitesPerBlock + threadIdx.x;
  const int mu = threadIdx.y;
  if (s >= g.V) return;
  int c[4], par;
  cb_coords(g, s, c, par);
  const uint32_t lex = (uint32_t)(c[0] + g.L[0] * (c[1] + g.L[1] * (c[2] + g.L[2] * c[3])));
  R z[12];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    uint32_t ctr[4] = {lex * 4u + (uint32_t)mu, draw, 5u, (uint32_t)q};
    Philox::rounds(ctr, k0, k1);
    box_muller<R>(ctr[0], ctr[1], z[4 * q + 0], z[4 * q + 1]);
    box_muller<R>(ctr[2], ctr[3], z[4 * q + 2], z[4 * q + 3]);
  }
  M3<R> u;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    u.e[0][j] = cx<R>(z[2 * j], z[2 * j + 1]);
    u.e[1][j] = cx<R>(z[6 + 2 * j], z[6 + 2 * j + 1]);
  }
  reunitarize(u);
  U.store(mu, s, u);
}

template <typename R, int NC>
__global__ void __launch_bounds__(256) reunitarize_kernel(Gauge<R, NC> U, int V) {
  const int s = blockIdx.x * kSitesPerBlock + threadIdx.x;
  const int mu = threadIdx.y;
  if (s >= V) return;
  M3<R> u = U.load(mu, s);
  reunitarize(u);
  U.store(mu, s, u);
}

constexpr int kEnergyThreads = 256;

// Per-site energies, one thread per site (blocks of 128 half-sites of both
// parities), block partial sums in the per-site value type A (double-float
// for FP32 fields: GB300's FP64 unit made the FP64 block tree and per-site
// arithmetic most of this kernel's time).
template <typename R>
using EnergyAcc =
    typename std::conditional<std::is_same<R, float>::value || std::is_same<R, DF>::value, DF, double>::type;

// Blocks of blockDim.x / 2 half-sites of both parities, or on small lattices
// of one warp, 32 half-sites of one parity.  The last block to finish (ticket,
// which it sets back to 0) adds the blocks' sums in block order into out[3].
template <typename R, int NC>
__global__ void __launch_bounds__(kEnergyThreads, (std::is_same<R, float>::value ? 2 : 1))
    energy_kernel(Gauge<R, NC> U, Mom<R> P, Geom g, EnergyAcc<R> beta6, EnergyAcc<R> beta3, int mode,
                  EnergyAcc<R>* __restrict__ h0, double* __restrict__ partial,
                  const EnergyAcc<R>* __restrict__ sg_in, EnergyAcc<R>* __restrict__ sg_out,
                  unsigned* __restrict__ ticket, double* __restrict__ out) {
  using A = EnergyAcc<R>;
  A v[3] = {A(0), A(0), A(0)};  // S_G, T, dh
  const bool narrow = blockDim.x == 32;
  const int H = narrow ? 32 : (int)blockDim.x >> 1;
  const int par = narrow ? blockIdx.x & 1 : (int)threadIdx.x >= H;
  const int i = (int)(narrow ? blockIdx.x >> 1 : blockIdx.x) * H + (int)threadIdx.x - (narrow ? 0 : par * H);
  if (i < g.Vh) site_energy(U, P, g, par * g.Vh + i, beta6, beta3, mode, h0, v, sg_in, sg_out);
  if constexpr (std::is_same<A, DF>::value) block_reduce_store_df<3>(v, partial, gridDim.x);
  else block_reduce_store<3>(v, partial, gridDim.x);
  __shared__ int last;
  if (threadIdx.x == 0) {  // the thread that has stored the block's sums
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  __shared__ double sh[3][8];
  const int n = gridDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double x[3] = {0.0, 0.0, 0.0};
#pragma unroll 4
  for (int b = threadIdx.x; b < n; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] += __ldcg(partial + (size_t)k * n + b);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x[k] += __shfl_down_sync(0xffffffffu, x[k], o);
    if (lane == 0) sh[k][warp] = x[k];
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[threadIdx.x][w];
    out[threadIdx.x] = t;
  }
  if (threadIdx.x == 0) *ticket = 0u;
}

__global__ void __launch_bounds__(1024) reduce_kernel(const double* __restrict__ partial, int nblocks,
                                                      int nv, double* __restrict__ out,
                                                      int accumulate) {
  __shared__ double sh[32];
  for (int k = 0; k < nv; ++k) {
    double x = 0.0;
    for (int i = threadIdx.x; i < nblocks; i += blockDim.x) x += partial[(size_t)k * nblocks + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
      x = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) out[k] = accumulate ? out[k] + x : x;
    }
    __syncthreads();
  }
}

template <typename R>
__global__ void __launch_bounds__(256) refresh_momenta_kernel(Mom<R> P, Geom g, uint32_t k0,
                                                              uint32_t k1, uint32_t draw) {
  const int s = blockIdx.x * kSitesPerBlock + threadIdx.x;
  const int mu = threadIdx.y;
  if (s >= g.V) return;
  refresh_link(P, g, s, mu, k0, k1, draw, 0u);
}

template <typename R, int NC>
__global__ void gauge_to_device_kernel(const double* __restrict__ canon, Gauge<R, NC> U, Geom g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // (lex, mu)
  if (i >= 4 * g.V) return;
  const int lex = i >> 2, mu = i & 3;
  int c[4];
  int r = lex;
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
  const int s = cb_index(g, c);
  M3<R> m;
  const double* src = canon + (size_t)i * 18;
#pragma unroll
  for (int k = 0; k < 9; ++k) m.e[k / 3][k % 3] = cx<R>(R(src[2 * k]), R(src[2 * k + 1]));
  U.store(mu, s, m);
}

template <typename R, int NC>
__global__ void gauge_to_canon_kernel(Gauge<R, NC> U, double* __restrict__ canon, Geom g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 4 * g.V) return;
  const int lex = i >> 2, mu = i & 3;
  int c[4];
  int r = lex;
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
  const M3<R> m = U.load(mu, cb_index(g, c));
  double* dst = canon + (size_t)i * 18;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    dst[2 * k] = double(m.e[k / 3][k % 3].re);
    dst[2 * k + 1] = double(m.e[k / 3][k % 3].im);
  }
}

template <typename R, typename T>
__global__ void mom_to_device_kernel(const T* __restrict__ canon, Mom<R> P, Geom g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 4 * g.V) return;
  const int lex = i >> 2, mu = i & 3;
  int c[4];
  int r = lex;
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
  R p[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) p[k] = R(canon[(size_t)i * 8 + k]);
  P.store(mu, cb_index(g, c), p);
}

template <typename R>
__global__ void mom_to_canon_kernel(Mom<R> P, double* __restrict__ canon, Geom g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 4 * g.V) return;
  const int lex = i >> 2, mu = i & 3;
  int c[4];
  int r = lex;
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
  R p[8];
  P.load(mu, cb_index(g, c), p);
#pragma unroll
  for (int k = 0; k < 8; ++k) canon[(size_t)i * 8 + k] = double(p[k]);
}

// ---------------------------------------------------------------------------
// Launchers.
template <typename R, int NC>
static Gauge<R, NC> gauge_of(const void* p, int V) {
  Gauge<R, NC> u;
  u.p = const_cast<void*>(p);
  u.V = V;
  return u;
}
template <typename R>
static Mom<R> mom_of(const void* p, int V) {
  Mom<R> m;
  m.p = const_cast<void*>(p);
  m.V = V;
  return m;
}

static inline dim3 link_grid(int V) { return dim3((V + kSitesPerBlock - 1) / kSitesPerBlock); }
static inline dim3 link_block() { return dim3(kSitesPerBlock, 4); }

template <int NC>
static cudaError_t launch_staple_force(const GeomH& gh, int mode, const ForceArgs& a, cudaStream_t st) {
  if constexpr (kForceSharedT<float, NC> && FG_FORCE_CARVEOUT > 0) {
    // keep the L1 share of the unified L1/shared storage as large as the
    // staple-product slots allow: the kernel's neighbour loads live in L1.
    // A preference only (once per process, thread-safe static initialisation);
    // a refusal leaves the driver's choice and is not an error.
    static const bool carved = [] {
      const cudaFuncAttribute a = cudaFuncAttributePreferredSharedMemoryCarveout;
      cudaFuncSetAttribute(staple_force_kernel<NC, FM_STORE>, a, FG_FORCE_CARVEOUT);
      cudaFuncSetAttribute(staple_force_kernel<NC, FM_KICK>, a, FG_FORCE_CARVEOUT);
      cudaFuncSetAttribute(staple_force_kernel<NC, FM_KICK_DRIFT>, a, FG_FORCE_CARVEOUT);
      cudaFuncSetAttribute(staple_force_kernel<NC, FM_DISPLACE>, a, FG_FORCE_CARVEOUT);
      cudaGetLastError();
      return true;
    }();
    (void)carved;
  }
  const Geom g = to_dev(gh);
  const int V = g.V;
  auto U = gauge_of<float, NC>(a.U, V);
  auto P = mom_of<float>(a.P, V);
  auto F = mom_of<float>(a.F, V);
  auto FF = mom_of<float>(a.FF, V);
  auto Ub = gauge_of<float, NC>(a.Ubase, V);
  auto Uo = gauge_of<float, NC>(a.Uout, V);
  const bool kick = mode == FM_KICK || mode == FM_KICK_DRIFT;
  const KickPair k = kick ? a.pair : KickPair{float(a.beta / 6.0), 0.0f, float(a.ffw == 0.0 ? 1.0 : a.ffw)};
  const int nb = 2 * ((g.Vh + kStapleSites - 1) / kStapleSites);
#define FG_FORCE(M)                                                                                          \
  staple_force_kernel<NC, M><<<nb, dim3(kStapleSites, 4), 0, st>>>(U, P, F, FF, Ub, Uo, g, k.a, k.b,        \
                                                                  a.drift.x, a.drift.y, float(a.cdisp), a.reunit, k.w)
  switch (mode) {
    case FM_STORE: FG_FORCE(FM_STORE); break;
    case FM_KICK: FG_FORCE(FM_KICK); break;
    case FM_KICK_DRIFT: FG_FORCE(FM_KICK_DRIFT); break;
    case FM_DISPLACE: FG_FORCE(FM_DISPLACE); break;
    default: return cudaErrorInvalidValue;
  }
#undef FG_FORCE
  return cudaGetLastError();
}

void fill_chain(void* dst, const GeomH& gh, double beta, long long goff, long long moff, long long woff,
                long long soff) {
  ChainDesc* cd = (ChainDesc*)dst;
  cd->g = to_dev(gh);
  cd->goff = goff; cd->moff = moff; cd->woff = woff; cd->soff = soff;
  cd->beta = beta;
  cd->beta6 = beta / 6.0;
  cd->beta6_hi = (float)cd->beta6;
  cd->beta6_lo = (float)(cd->beta6 - (double)cd->beta6_hi);
  cd->tile0 = cd->ntiles = 0;
}
size_t chain_bytes() { return sizeof(ChainDesc); }

template <typename R, int NC>
cudaError_t launch_plaquettes(const ForceRows& r, const void* U, void* W, cudaStream_t st) {
  const long long warps = 12LL * r.nrows;
  const int w = warps_per_block(warps, kForceThreads / 32);
  plaquette_kernel<R, NC><<<(unsigned)((warps + w - 1) / w), 32 * w, 0, st>>>(r, (char*)U, (char*)W);
  return cudaGetLastError();
}

template <typename R, int NC>
cudaError_t launch_unitarity(const ForceRows& r, const void* U, double* flag, int stride, cudaStream_t st) {
  const long long warps = 8LL * r.nrows;
  const int w = warps_per_block(warps, kForceThreads / 32);
  unitarity_kernel<R, NC><<<(unsigned)((warps + w - 1) / w), 32 * w, 0, st>>>(r, (char*)U, R(kUnitaryWithin<R>), flag,
                                                                             stride);
  return cudaGetLastError();
}

template <typename R, int NC>
static cudaError_t launch_link_force(const ForceRows& r, int mode, const ForceArgs& a, cudaStream_t st) {
  const R ckick = R(a.ckick), ffw = R(a.ffw == 0.0 ? 1.0 : a.ffw), cdrift = R(a.cdrift);
  const long long warps = 8LL * r.nrows;
  const int w = warps_per_block(warps, kForceThreads / 32);
  const unsigned nb = (unsigned)((warps + w - 1) / w);
#define FG_FORCE(M)                                                                                                   \
  do {                                                                                                                \
    if (a.W != nullptr)                                                                                               \
      link_force_kernel<R, NC, M><<<nb, 32 * w, 0, st>>>(r, (char*)a.U, (char*)a.W, (char*)a.P, (char*)a.F, (char*)a.FF, \
                                                         (char*)a.Ubase, (char*)a.Uout, ckick, cdrift, R(0), R(a.cdisp), \
                                                         a.reunit, ffw);                                              \
    else                                                                                                              \
      staple_rows_kernel<R, NC, M><<<nb, 32 * w, 0, st>>>(r, (char*)a.U, (char*)a.P, (char*)a.F, (char*)a.FF,         \
                                                          (char*)a.Ubase, (char*)a.Uout, ckick, cdrift, R(0), R(a.cdisp), \
                                                          a.reunit, ffw);                                             \
  } while (0)
  switch (mode) {
    case FM_STORE: FG_FORCE(FM_STORE); break;
    case FM_KICK: FG_FORCE(FM_KICK); break;
    case FM_KICK_DRIFT: FG_FORCE(FM_KICK_DRIFT); break;
    case FM_DISPLACE: FG_FORCE(FM_DISPLACE); break;
    default: return cudaErrorInvalidValue;
  }
#undef FG_FORCE
  return cudaGetLastError();
}

template <typename R, int NC>
cudaError_t launch_gauge_force(const GeomH& gh, const ForceRows& rows, int mode, const ForceArgs& a,
                               cudaStream_t st) {
  if constexpr (kPlaquetteForce<R>) return launch_link_force<R, NC>(rows, mode, a, st);
  else return launch_staple_force<NC>(gh, mode, a, st);
}

template <typename R, int NC>
cudaError_t launch_drift(const GeomH& gh, const void* Uin, const void* P, void* Uout, double c,
                         int reunit, cudaStream_t st) {
  const long long warps = 4LL * ((gh.V + 31) / 32);
  const int w = warps_per_block(warps, 8);
  R x = R(c), y = R(0);
  if constexpr (std::is_same<R, float>::value) {
    const DriftPair d = drift_pair(c);
    x = d.x;
    y = d.y;
  }
  drift_kernel<R, NC><<<(unsigned)((warps + w - 1) / w), 32 * w, 0, st>>>(
      gauge_of<R, NC>(Uin, gh.V), mom_of<R>(P, gh.V), gauge_of<R, NC>(Uout, gh.V), gh.V, x, y, reunit);
  return cudaGetLastError();
}

template <typename R, int NC>
cudaError_t launch_unit_links(const GeomH& gh, void* U, cudaStream_t st) {
  unit_links_kernel<R, NC><<<link_grid(gh.V), link_block(), 0, st>>>(gauge_of<R, NC>(U, gh.V), gh.V);
  return cudaGetLastError();
}

template <typename R, int NC>
cudaError_t launch_random_links(const GeomH& gh, void* U, uint64_t seed, uint32_t draw, cudaStream_t st) {
  random_links_kernel<R, NC><<<link_grid(gh.V), link_block(), 0, st>>>(gauge_of<R, NC>(U, gh.V), to_dev(gh),
                                                                       (uint32_t)seed, (uint32_t)(seed >> 32), draw);
  return cudaGetLastError();
}

template <typename R, int NC>
cudaError_t launch_reunitarize(const GeomH& gh, void* U, cudaStream_t st) {
  reunitarize_kernel<R, NC><<<link_grid(gh.V), link_block(), 0, st>>>(gauge_of<R, NC>(U, gh.V), gh.V);
  return cudaGetLastError();
}

int energy_blocks(const GeomH& gh) {
  const int t = 32 * warps_per_block((gh.V + 31) / 32, kEnergyThreads / 32);
  return t == 32 ? 2 * ((gh.Vh + 31) / 32) : (gh.Vh + t / 2 - 1) / (t / 2);
}

template <typename R, int NC>
cudaError_t launch_energy(const GeomH& gh, const void* U, const void* P, double beta, int mode,
                          double* h0, double* partial, unsigned* ticket, double* out, cudaStream_t st,
                          const double* sg_in, double* sg_out) {
  const int t = 32 * warps_per_block((gh.V + 31) / 32, kEnergyThreads / 32);
  // the per-site arrays are 8 bytes a site: doubles, or double-floats for FP32 fields
  using A = EnergyAcc<R>;
  static_assert(sizeof(A) == sizeof(double), "per-site slot size");
  energy_kernel<R, NC><<<energy_blocks(gh), t, 0, st>>>(
      gauge_of<R, NC>(U, gh.V), mom_of<R>(P, gh.V), to_dev(gh), A(6.0 * beta), A(beta / 3.0), mode,
      reinterpret_cast<A*>(h0), partial, reinterpret_cast<const A*>(sg_in), reinterpret_cast<A*>(sg_out), ticket, out);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const double* partial, int nblocks, int nv, double* out, int accumulate,
                          cudaStream_t st) {
  reduce_kernel<<<1, 1024, 0, st>>>(partial, nblocks, nv, out, accumulate);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_refresh_momenta(const GeomH& gh, void* P, uint64_t seed, uint32_t draw,
                                   cudaStream_t st) {
  refresh_momenta_kernel<R><<<link_grid(gh.V), link_block(), 0, st>>>(
      mom_of<R>(P, gh.V), to_dev(gh), (uint32_t)seed, (uint32_t)(seed >> 32), draw);
  return cudaGetLastError();
}

template <typename R, int NC>
cudaError_t launch_gauge_to_device(const GeomH& gh, const double* canon, void* U, cudaStream_t st) {
  gauge_to_device_kernel<R, NC><<<(4 * gh.V + 255) / 256, 256, 0, st>>>(canon, gauge_of<R, NC>(U, gh.V),
                                                                       to_dev(gh));
  return cudaGetLastError();
}
template <typename R, int NC>
cudaError_t launch_gauge_to_canon(const GeomH& gh, const void* U, double* canon, cudaStream_t st) {
  gauge_to_canon_kernel<R, NC><<<(4 * gh.V + 255) / 256, 256, 0, st>>>(gauge_of<R, NC>(U, gh.V), canon,
                                                                      to_dev(gh));
  return cudaGetLastError();
}
template <typename R>
cudaError_t launch_mom_to_device(const GeomH& gh, const double* canon, void* P, cudaStream_t st) {
  mom_to_device_kernel<R, double><<<(4 * gh.V + 255) / 256, 256, 0, st>>>(canon, mom_of<R>(P, gh.V), to_dev(gh));
  return cudaGetLastError();
}
template <typename R>
cudaError_t launch_mom_to_canon(const GeomH& gh, const void* P, double* canon, cudaStream_t st) {
  mom_to_canon_kernel<R><<<(4 * gh.V + 255) / 256, 256, 0, st>>>(mom_of<R>(P, gh.V), canon, to_dev(gh));
  return cudaGetLastError();
}

// P -= c FF (kick with a force computed elsewhere: the pseudofermion force of
// a two-level integrator's outer kicks).
template <typename R>
__global__ void __launch_bounds__(256) kick_ff_kernel(Mom<R> P, Mom<R> FF, int V, R a, R b) {
  const int s = blockIdx.x * kSitesPerBlock + threadIdx.x;
  const int mu = threadIdx.y;
  if (s >= V) return;
  R p[8], f[8];
  P.load(mu, s, p);
  FF.load(mu, s, f);
#pragma unroll
  for (int k = 0; k < 8; ++k) p[k] = fma(-b, a * f[k], p[k]);
  P.store(mu, s, p);
}
template <typename R>
cudaError_t launch_kick_ff(const GeomH& gh, void* P, const void* FF, double c, cudaStream_t st) {
  R a = R(1.0f), b = R(c);
  if constexpr (std::is_same<R, float>::value) {
    const KickPair k = kick_pair(c);
    a = k.a;
    b = k.b;
  }
  kick_ff_kernel<R><<<link_grid(gh.V), link_block(), 0, st>>>(mom_of<R>(P, gh.V), mom_of<R>(FF, gh.V), gh.V, a, b);
  return cudaGetLastError();
}
template cudaError_t launch_kick_ff<double>(const GeomH&, void*, const void*, double, cudaStream_t);
template cudaError_t launch_kick_ff<float>(const GeomH&, void*, const void*, double, cudaStream_t);
template cudaError_t launch_kick_ff<DF>(const GeomH&, void*, const void*, double, cudaStream_t);

template cudaError_t launch_unitarity<double, 9>(const ForceRows&, const void*, double*, int, cudaStream_t);
template cudaError_t launch_unitarity<double, 6>(const ForceRows&, const void*, double*, int, cudaStream_t);
template cudaError_t launch_unitarity<DF, 9>(const ForceRows&, const void*, double*, int, cudaStream_t);
template cudaError_t launch_unitarity<DF, 6>(const ForceRows&, const void*, double*, int, cudaStream_t);
template cudaError_t launch_plaquettes<double, 9>(const ForceRows&, const void*, void*, cudaStream_t);
template cudaError_t launch_plaquettes<double, 6>(const ForceRows&, const void*, void*, cudaStream_t);
template cudaError_t launch_plaquettes<DF, 9>(const ForceRows&, const void*, void*, cudaStream_t);
template cudaError_t launch_plaquettes<DF, 6>(const ForceRows&, const void*, void*, cudaStream_t);

#define FG_INST_RNC(R, NC)                                                                          \
  template cudaError_t launch_gauge_force<R, NC>(const GeomH&, const ForceRows&, int, const ForceArgs&,   \
                                                 cudaStream_t);                                   \
  template cudaError_t launch_drift<R, NC>(const GeomH&, const void*, const void*, void*, double,   \
                                           int, cudaStream_t);                                      \
  template cudaError_t launch_reunitarize<R, NC>(const GeomH&, void*, cudaStream_t);                \
  template cudaError_t launch_unit_links<R, NC>(const GeomH&, void*, cudaStream_t);                 \
  template cudaError_t launch_random_links<R, NC>(const GeomH&, void*, uint64_t, uint32_t, cudaStream_t); \
  template cudaError_t launch_energy<R, NC>(const GeomH&, const void*, const void*, double, int,    \
                                            double*, double*, unsigned*, double*, cudaStream_t,     \
                                            const double*, double*);                                \
  template cudaError_t launch_gauge_to_device<R, NC>(const GeomH&, const double*, void*,            \
                                                     cudaStream_t);                                 \
  template cudaError_t launch_gauge_to_canon<R, NC>(const GeomH&, const void*, double*, cudaStream_t);

FG_INST_RNC(double, 9)
FG_INST_RNC(double, 6)
FG_INST_RNC(float, 9)
FG_INST_RNC(float, 6)
FG_INST_RNC(DF, 9)
FG_INST_RNC(DF, 6)

template cudaError_t launch_refresh_momenta<double>(const GeomH&, void*, uint64_t, uint32_t, cudaStream_t);
template cudaError_t launch_refresh_momenta<float>(const GeomH&, void*, uint64_t, uint32_t, cudaStream_t);
template cudaError_t launch_refresh_momenta<DF>(const GeomH&, void*, uint64_t, uint32_t, cudaStream_t);
template cudaError_t launch_mom_to_device<double>(const GeomH&, const double*, void*, cudaStream_t);
template cudaError_t launch_mom_to_device<float>(const GeomH&, const double*, void*, cudaStream_t);
template cudaError_t launch_mom_to_device<DF>(const GeomH&, const double*, void*, cudaStream_t);
template <typename R>
cudaError_t launch_mom_to_device_f32(const GeomH& gh, const float* canon, void* P, cudaStream_t st) {
  mom_to_device_kernel<R, float><<<(4 * gh.V + 255) / 256, 256, 0, st>>>(canon, mom_of<R>(P, gh.V), to_dev(gh));
  return cudaGetLastError();
}
template cudaError_t launch_mom_to_device_f32<double>(const GeomH&, const float*, void*, cudaStream_t);
template cudaError_t launch_mom_to_device_f32<float>(const GeomH&, const float*, void*, cudaStream_t);
template cudaError_t launch_mom_to_device_f32<DF>(const GeomH&, const float*, void*, cudaStream_t);
template cudaError_t launch_mom_to_canon<double>(const GeomH&, const void*, double*, cudaStream_t);
template cudaError_t launch_mom_to_canon<float>(const GeomH&, const void*, double*, cudaStream_t);
template cudaError_t launch_mom_to_canon<DF>(const GeomH&, const void*, double*, cudaStream_t);

// FP32 FMA throughput probe: eight independent FMA chains per thread, 16
// FMAs of each per loop trip, one store per thread so nothing is dropped.
// a <- a b + c with b = 1 - 1e-4 and c = 1e-4 stays near 1 (no overflow or
// subnormals).
__global__ void __launch_bounds__(256) fma_rate_kernel(float* __restrict__ out, int iters, float b, float c) {
  float a[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) a[k] = 0.5f + 0.01f * float(k) + 1e-6f * float(threadIdx.x);
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int u = 0; u < 16; ++u)
#pragma unroll
      for (int k = 0; k < 8; ++k) a[k] = fmaf(a[k], b, c);
  }
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < 8; ++k) s += a[k];
  out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

cudaError_t launch_fma_rate(float* out, int blocks, int iters, cudaStream_t st) {
  fma_rate_kernel<<<blocks, 256, 0, st>>>(out, iters, 1.0f - 1e-4f, 1e-4f);
  return cudaGetLastError();
}

}  // namespace fg
