// Host-side launchers of the device kernels (implemented in gauge.cu and
// fermion.cu, used by the runtime in fg_lattice.cu).  Every launcher enqueues
// on `st` and returns the cudaError_t of the launch.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstdlib>
#include <type_traits>

namespace fg {

struct GeomH {
  int L[4];
  int Lxh, Vh, V;
  bool shared = false;   // the lattice shares the GPU with others (fg_set_shared)
};

// Fused gauge-force kernel modes.
enum ForceMode {
  FM_STORE = 0,       // F_out = F(U) (+ FF)
  FM_KICK = 1,        // P -= ckick F(U)
  FM_KICK_DRIFT = 2,  // P -= ckick F(U); U_out = exp(i cdrift P) U_base
  FM_DISPLACE = 3     // U_out = exp(-i cdisp F(U)) U
};

// FP32 kicks P -= k F + c FF are formed as f = a F + w FF, P -= b f.  A
// coefficient rounded to FP32 is an error of one sign: k = 1/48 comes out too
// strong by 3e-8 on every link, and by more because products with its periodic
// digits often lie just at the middle between two momenta, so the trajectory
// conserves T + (1 + e) S and dH is off by e times what S has gained, in
// proportion to the volume.  a and b are two FP32 numbers whose product is k to
// some 1e-10 (7e-9 at worst of 20000 coefficients; with b w = c beside it some
// 1e-9, 1.4e-8 at worst), with digits of no pattern: a is taken near the golden
// ratio.  FG, dt = 1/8, from links still relaxing: dH off by
// 5.0e-3 (32^4) and 5e-4 (16^4), with rounded coefficients 0.112 and 6.3e-3.
// The device executes the same operations (coefficients with low parts, added
// by compensated arithmetic, did as well and took 1.5% of a 32^4 trajectory).
struct KickPair {
  float a, b, w;
};
inline KickPair kick_pair(double k, double c = 0.0) {
  // for coefficients out of FP32's range, whose products say so
  KickPair best = k != 0.0 ? KickPair{1.0f, (float)k, (float)(c / k)} : KickPair{0.0f, (float)c, c != 0.0 ? 1.0f : 0.0f};
  double least = 1e300;
  const int n = c != 0.0 ? 1024 : 128;
  for (int i = 0; i < n; ++i) {
    const double x = (double)(float)(1.6180339887498949 * (1.0 + i * 0x1p-18));
    const float b = (float)((k != 0.0 ? k : c) / x);
    double e = std::fabs(x * b - k);
    float w = 0.0f;
    if (c != 0.0) {
      w = (float)(c / b);
      e = std::fabs((double)w * b / c - 1.0);
      if (k != 0.0) e = std::fmax(e, std::fabs(x * b / k - 1.0));
    }
    if (e < least) {
      least = e;
      best = KickPair{k != 0.0 ? (float)x : 0.0f, b, w};
    }
  }
  return best;
}

// FP32 drifts by exp(i c P) likewise: the exponent is y sum_a (x p^a) lambda^a
// with x y = c / 2.
struct DriftPair {
  float x, y;
};
inline DriftPair drift_pair(double c) {
  const KickPair k = kick_pair(0.5 * c);
  return DriftPair{k.a, k.b};
}

struct ForceArgs {
  const void* U;       // links at which the force is evaluated
  const void* W;       // their plaquette field (launch_plaquettes), or null for the staple sums (FP32: unused)
  void* P;             // momenta
  void* F;             // force out (FM_STORE)
  const void* FF;      // extra force added to the gauge force (fermions) or nullptr
  const void* Ubase;   // drift base links (FM_KICK_DRIFT); may equal U
  void* Uout;          // output links (FM_KICK_DRIFT, FM_DISPLACE)
  double beta;
  double ckick, cdrift, cdisp;
  KickPair pair;       // FP32 kicks, in place of ckick, beta and ffw
  DriftPair drift;     // FP32 drifts, in place of cdrift
  double ffw;          // weight of FF relative to the gauge force (0 is treated as 1)
  int reunit;
};

// Whether the force of links in precision R can be formed by plaquettes (two
// launches), or always by staples (one).
template <typename R>
constexpr bool kPlaquetteForce = !std::is_same<R, float>::value;

inline bool plaquettes_off() {
  const char* e = std::getenv("FG_PLAQUETTES");
  return e && e[0] == '0';
}

// The lattices of an FP64 or double-float force launch, cut into rows of 32
// half-sites.
struct ForceRows {
  const void* chains;     // device array of lattice descriptions (fill_chain)
  const int2* rows;       // lattice and first half-site of each row, or null for all rows of one lattice
  int nrows;
};
void fill_chain(void* dst, const GeomH& g, double beta, long long goff, long long moff, long long woff,
                long long soff);
size_t chain_bytes();

// The plaquette field of links U into W (6 x 8 reals a site), which the force
// launch that follows reads.
template <typename R, int NC>
cudaError_t launch_plaquettes(const ForceRows& rows, const void* U, void* W, cudaStream_t st);
// flag[stride * lattice] = 1.0 for every lattice of `rows` with links too far
// from unitary for the plaquette form (untouched otherwise).
template <typename R, int NC>
cudaError_t launch_unitarity(const ForceRows& rows, const void* U, double* flag, int stride, cudaStream_t st);
// `rows` is used in FP64 and double-float, `g` in FP32.
template <typename R, int NC>
cudaError_t launch_gauge_force(const GeomH& g, const ForceRows& rows, int mode, const ForceArgs& a, cudaStream_t st);

// P -= c FF on every link (a kick with an externally computed force).
template <typename R>
cudaError_t launch_kick_ff(const GeomH& g, void* P, const void* FF, double c, cudaStream_t st);

// Closed-form force gradient (forcegrad.cu): dU = i F U on every link
// (dU stored with NC = 9); G = derivative of the gauge force along dU, plus
// FFt if not null; P -= c (F - shift G).
template <typename R, int NC>
cudaError_t launch_tangent_links(const GeomH& g, const void* U, const void* F, void* dU, cudaStream_t st);
template <typename R, int NC>
cudaError_t launch_force_tangent(const GeomH& g, const void* U, const void* dU, void* G, const void* FFt,
                                 double beta, cudaStream_t st);
template <typename R>
cudaError_t launch_kick_fg(const GeomH& g, void* P, const void* F, const void* G, double c, double shift,
                           cudaStream_t st);

// U_out = exp(i c P) U_in on every link (U_out may equal U_in).
template <typename R, int NC>
cudaError_t launch_drift(const GeomH& g, const void* Uin, const void* P, void* Uout, double c,
                         int reunit, cudaStream_t st);

// Every link = identity (cold start).
template <typename R, int NC>
cudaError_t launch_unit_links(const GeomH& g, void* U, cudaStream_t st);
// FP32 FMA throughput probe: `blocks` blocks of 256 threads, each running
// 8 chains x 16 x iters FMAs; out holds blocks x 256 floats.
cudaError_t launch_fma_rate(float* out, int blocks, int iters, cudaStream_t st);

// Haar-random SU(3) links (device hot start).
template <typename R, int NC>
cudaError_t launch_random_links(const GeomH& g, void* U, uint64_t seed, uint32_t draw, cudaStream_t st);

template <typename R, int NC>
cudaError_t launch_reunitarize(const GeomH& g, void* U, cudaStream_t st);

// Per-site energy h(x) = T(x) + S_G(x) (T = 0 if P is null).  mode 0: also
// store h0[x] = h(x); mode 1: also sum h(x) - h0[x]; mode 2: sums only.  The
// sums of (S_G, T, dh) go to out[3] through 3 x energy_blocks block sums in
// `partial` and the counter *ticket (0 before, 0 after).
// sg_in (optional): per-site S_G of these links stored earlier, used instead
// of the plaquettes; sg_out (optional): per-site S_G stored for later.
int energy_blocks(const GeomH& g);
template <typename R, int NC>
cudaError_t launch_energy(const GeomH& g, const void* U, const void* P, double beta, int mode,
                          double* h0, double* partial, unsigned* ticket, double* out, cudaStream_t st,
                          const double* sg_in = nullptr, double* sg_out = nullptr);

// out[k] += sum_b partial[k][b] for k < nv (fixed order, one block).  If
// `accumulate` is 0 the sums overwrite out[k].
cudaError_t launch_reduce(const double* partial, int nblocks, int nv, double* out, int accumulate,
                          cudaStream_t st);

// Unit-Gaussian momenta from Philox-4x32-10 keyed by seed, counter (link, draw).
template <typename R>
cudaError_t launch_refresh_momenta(const GeomH& g, void* P, uint64_t seed, uint32_t draw,
                                   cudaStream_t st);

// Layout conversion between the canonical FP64 host order and device SoA.
template <typename R, int NC>
cudaError_t launch_gauge_to_device(const GeomH& g, const double* canon, void* U, cudaStream_t st);
template <typename R, int NC>
cudaError_t launch_gauge_to_canon(const GeomH& g, const void* U, double* canon, cudaStream_t st);
template <typename R>
cudaError_t launch_mom_to_device(const GeomH& g, const double* canon, void* P, cudaStream_t st);
// The same from canonical FP32 momenta.
template <typename R>
cudaError_t launch_mom_to_device_f32(const GeomH& g, const float* canon, void* P, cudaStream_t st);
template <typename R>
cudaError_t launch_mom_to_canon(const GeomH& g, const void* P, double* canon, cudaStream_t st);

// Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC11), usable on host and device.
struct Philox {
  static inline __host__ __device__ void mulhilo(uint32_t a, uint32_t b, uint32_t& hi, uint32_t& lo) {
    const uint64_t p = (uint64_t)a * (uint64_t)b;
    hi = (uint32_t)(p >> 32);
    lo = (uint32_t)p;
  }
  static inline __host__ __device__ void rounds(uint32_t c[4], uint32_t k0, uint32_t k1) {
    for (int r = 0; r < 10; ++r) {
      uint32_t hi0, lo0, hi1, lo1;
      mulhilo(0xD2511F53u, c[0], hi0, lo0);
      mulhilo(0xCD9E8D57u, c[2], hi1, lo1);
      const uint32_t n0 = hi1 ^ c[1] ^ k0;
      const uint32_t n2 = hi0 ^ c[3] ^ k1;
      c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
  }
};

}  // namespace fg
