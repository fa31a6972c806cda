// hlb_common.cuh — device-side building blocks of the D3Q19 sparse-lattice
// solver: velocity tables, shifted-population storage traits, link records,
// kernel parameters, and the per-site gather (streaming + boundaries) and
// BGK collision shared by the forward, readback and adjoint kernels.
//
// Method (arXiv 2202.11770): Section 2.2 (D3Q19, Eqs. 3a-3b, 4-6),
// Section 2.3 (bounce-back walls, Ladd velocity iolets, ghost-density
// pressure iolets), Section 3.2.3 (structure-of-arrays populations).
// Streaming is done as a pull (gather) through the streaming-index table,
// the ordering the paper's future-work list (Section 7, item 3) expects to
// be faster than its push kernels.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hlb {

constexpr int Q = 19;

// Velocity set (Section 2.2) in the order documented in hemegb.h.
__host__ __device__ constexpr int cx(int i) {
  constexpr int t[Q] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
  return t[i];
}
__host__ __device__ constexpr int cy(int i) {
  constexpr int t[Q] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
  return t[i];
}
__host__ __device__ constexpr int cz(int i) {
  constexpr int t[Q] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
  return t[i];
}
// Opposite pairs are adjacent: 1<->2, 3<->4, ..., 17<->18.
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
// Weights 1/3, 1/18, 1/36 (Section 2.2).
template <typename R>
__host__ __device__ constexpr R wgt(int i) {
  return i == 0 ? R(1) / R(3) : (i <= 6 ? R(1) / R(18) : R(1) / R(36));
}

// ---------------------------------------------------------------------------
// Storage traits: populations are stored shifted, h = f - w.
// ---------------------------------------------------------------------------
template <typename S> struct Real { using type = float; };
template <> struct Real<double> { using type = double; };

__device__ __forceinline__ float to_real(float v) { return v; }
__device__ __forceinline__ double to_real(double v) { return v; }
__device__ __forceinline__ float to_real(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_real(__half v) { return __half2float(v); }

template <typename S> __device__ __forceinline__ S from_real(float v);
template <> __device__ __forceinline__ float from_real<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_real<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}
template <> __device__ __forceinline__ __half from_real<__half>(float v) { return __float2half_rn(v); }
template <typename S> __device__ __forceinline__ S from_real(double v);
template <> __device__ __forceinline__ double from_real<double>(double v) { return v; }

// Programmatic dependent launch (sm_90 and later).  A step kernel lets the
// next kernel of its stream be scheduled as soon as all of its own blocks are
// resident (pdl_trigger), and waits for the previous kernel to complete, its
// memory visible, before it reads anything that kernel wrote (pdl_wait).  The
// next kernel's blocks then fill the SMs that the tail of this one frees,
// instead of waiting for the launch after it ends.  Without the launch
// attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Cached load of a population (read-only for the whole kernel).
template <typename S>
__device__ __forceinline__ typename Real<S>::type ldpop(const S* p) {
  return to_real(__ldg(p));
}
// Streaming store of a population (next read is a full sweep later).
template <typename S>
__device__ __forceinline__ void stpop(S* p, typename Real<S>::type v) {
  __stcs(p, from_real<S>(v));
}

// ---------------------------------------------------------------------------
// Boundary links and per-launch parameters.
// ---------------------------------------------------------------------------
// One record per (site, pull direction) whose source crosses an iolet.  In
// the device index table such a link carries the code -(2 + record index).
struct LinkRec {
  int32_t site;
  int8_t dir;      // pull direction j: the source x - c_j is beyond the iolet
  int8_t kind;     // 0 velocity, 1 pressure
  int16_t iolet;
  int32_t group;   // global amplitude group (velocity), -1 otherwise
  float coef_f;    // (float) coef, rounded on the host
  double coef;     // velocity: 6 w_j W(x_m) (c_j . n); pressure: unused
};
static_assert(sizeof(LinkRec) == 24, "LinkRec is 24 bytes");

constexpr int MAX_IOLETS = 128;

// Parameters are carried in double and rounded to the compute type at use,
// so that FP64 storage sees no FP32-rounded coefficient anywhere.
struct IoletParam {
  double nx, ny, nz;
  double val;  // velocity iolet: waveform factor w(t); pressure iolet: rho(t) - 1
  float nxf, nyf, nzf, valf;  // the same rounded to float on the host
};

struct StepParams {
  int64_t n;
  int64_t sn;           // row stride of the index table: n rounded up to a multiple of 4
  double omega;         // 1 / tau
  int32_t n_iolets;
  int32_t ladd_rho_one;
  int32_t ghost_full_u;
  float omegaf;         // (float) omega, rounded on the host: FP64 arithmetic is slow on GB300
                        // (1/64 of the FP32 rate), so FP32 kernels convert no double per thread
  uint64_t coupled[MAX_IOLETS / 64];  // bit k: iolet k's value lives in ioval[k] (Windkessel outlet)
  const double* ioval;                // device, [n_iolets]: rho - 1 of coupled outlets
  const float* ampf;                  // device, [amplitude groups]: the amplitudes rounded to float
  IoletParam io[MAX_IOLETS];
};
static_assert(MAX_IOLETS % 64 == 0, "coupling mask words");

// Division of a block number b < 2^31 by a fixed divisor d without an
// integer divide in the kernel: q = (b >> s) for d a power of two (m = 0),
// else q = umulhi(b, m) >> s with l = ceil(log2 d), m = ceil(2^(31+l) / d),
// s = l - 1, which is exact for all b < 2^31 (Granlund and Montgomery,
// "Division by invariant integers using multiplication", 1994: m d lies in
// [2^(31+l), 2^(31+l) + 2^l]).
struct BlockDiv {
  uint32_t d, m, s;
};
inline BlockDiv make_block_div(uint32_t d) {
  BlockDiv r{d, 0u, 0u};
  if ((d & (d - 1)) == 0) {
    while ((1u << r.s) < d) ++r.s;
    return r;
  }
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;  // ceil(log2 d)
  r.m = (uint32_t)((((uint64_t)1 << (31 + l)) + d - 1) / d);
  r.s = l - 1;
  return r;
}
__device__ __forceinline__ uint32_t block_div(uint32_t b, const BlockDiv& q) {
  return q.m == 0 ? (b >> q.s) : (__umulhi(b, q.m) >> q.s);
}

// How the iolet blocks of a step's grid lie among its bulk blocks.  The site
// list is cut into kSpread segments; the blocks of segment s are the grid's
// blocks [blk[s], blk[s + 1]), of which the iolet blocks number io[s] ..
// io[s + 1] - 1, evenly spaced.  An iolet site so runs at about the time that
// its neighbours in memory do: its 4 (2) bytes of a 32-byte sector join theirs
// in L2, where the same blocks spread over the whole grid wrote the sector to
// DRAM twice.  Block r of a segment is an iolet block when floor(r k / 2^32)
// steps from r to r + 1, k = ceil(2^32 iolet blocks / blocks).  segments = 1:
// the whole grid is segment 0 (no search).
constexpr int kSpread = 64;
struct IoletSpread {
  uint32_t segments, blk[kSpread + 1], io[kSpread + 1], k[kSpread];
};
// True for an iolet block, *number its number; else *number the bulk block's.
__device__ __forceinline__ bool spread_block(const IoletSpread& sp, uint32_t b, uint32_t* number) {
  int s = 0;
  if (sp.segments > 1) {
#pragma unroll
    for (int step = kSpread / 2; step > 0; step >>= 1)
      if (sp.blk[s + step] <= b) s += step;
  }
  const uint32_t r = b - sp.blk[s], before = __umulhi(r, sp.k[s]);
  const bool iolet = __umulhi(r + 1, sp.k[s]) != before;
  *number = iolet ? sp.io[s] + before : b - sp.io[s] - before;
  return iolet;
}

// Relaxation rate 1/tau in the arithmetic type of a kernel.
template <typename R> __device__ __forceinline__ R omega_of(const StepParams& p);
template <> __device__ __forceinline__ float omega_of<float>(const StepParams& p) { return p.omegaf; }
template <> __device__ __forceinline__ double omega_of<double>(const StepParams& p) { return p.omega; }

// Boundary value of iolet k for this launch: the host waveform, or for a
// Windkessel outlet the ghost density the device-side model last produced.
__device__ __forceinline__ double io_val(const StepParams& p, int k) {
  return ((p.coupled[k >> 6] >> (k & 63)) & 1ull) ? p.ioval[k] : p.io[k].val;
}

// Boundary data in the arithmetic type R of a kernel.  FP32 kernels read
// copies rounded to float on the host (or, for a Windkessel outlet's ghost
// density, once on the device): the value is the one R(x) would give, without
// a conversion from double per use (FP64 arithmetic runs at 1/64 of the FP32
// rate on GB300).
template <typename R> struct BC;
template <> struct BC<float> {
  static __device__ __forceinline__ float val(const StepParams& p, int k) {
    return ((p.coupled[k >> 6] >> (k & 63)) & 1ull) ? (float)p.ioval[k] : p.io[k].valf;
  }
  static __device__ __forceinline__ float coef(const LinkRec& L) { return L.coef_f; }
  static __device__ __forceinline__ float amp(const StepParams& p, const double*, int g) { return p.ampf[g]; }
  static __device__ __forceinline__ float nx(const IoletParam& q) { return q.nxf; }
  static __device__ __forceinline__ float ny(const IoletParam& q) { return q.nyf; }
  static __device__ __forceinline__ float nz(const IoletParam& q) { return q.nzf; }
};
template <> struct BC<double> {
  static __device__ __forceinline__ double val(const StepParams& p, int k) { return io_val(p, k); }
  static __device__ __forceinline__ double coef(const LinkRec& L) { return L.coef; }
  static __device__ __forceinline__ double amp(const StepParams&, const double* a, int g) { return a[g]; }
  static __device__ __forceinline__ double nx(const IoletParam& q) { return q.nx; }
  static __device__ __forceinline__ double ny(const IoletParam& q) { return q.ny; }
  static __device__ __forceinline__ double nz(const IoletParam& q) { return q.nz; }
};

// ---------------------------------------------------------------------------
// Moments and equilibrium in shifted form.
//   rho = 1 + drho, drho = sum h_i;  j = sum h_i c_i;  u = j / rho
//   f^eq_i - w_i = w_i (drho + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u.u))
// which is Eq. 4 with the factors 1/2 (cs2 = 1/3).
// ---------------------------------------------------------------------------
template <typename R>
struct Macro {
  R drho, rho, ux, uy, uz;
};

template <typename R>
__device__ __forceinline__ Macro<R> moments(const R* h) {
  R d = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    d += h[i];
    if (cx(i)) jx += cx(i) > 0 ? h[i] : -h[i];
    if (cy(i)) jy += cy(i) > 0 ? h[i] : -h[i];
    if (cz(i)) jz += cz(i) > 0 ? h[i] : -h[i];
  }
  Macro<R> m;
  m.drho = d;
  m.rho = R(1) + d;
  R inv = R(1) / m.rho;
  m.ux = jx * inv;
  m.uy = jy * inv;
  m.uz = jz * inv;
  return m;
}

template <typename R>
__device__ __forceinline__ R cdotu(int i, R ux, R uy, R uz) {
  R s = R(0);
  if (cx(i)) s += cx(i) > 0 ? ux : -ux;
  if (cy(i)) s += cy(i) > 0 ? uy : -uy;
  if (cz(i)) s += cz(i) > 0 ? uz : -uz;
  return s;
}

__device__ __forceinline__ float fmadd(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmadd(double a, double b, double c) { return __fma_rn(a, b, c); }

// Sums of products, whose products the compiler may contract either way.  Its
// choice differed between kernels, so the boundary values write the fused
// operations out: every path gives the same bits.
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double fmul(double a, double b) { return __dmul_rn(a, b); }
template <typename R>
__device__ __forceinline__ R dot3(R ax, R ay, R az, R bx, R by, R bz) {
  return fmadd(az, bz, fmadd(ax, bx, fmul(ay, by)));
}
// Ghost value w (drho + rho (3 cu + 4.5 cu^2 - 1.5 u.u)) of a pressure iolet.
template <typename R>
__device__ __forceinline__ R ghost_heq(R w, R drho, R cu, R uu) {
  const R t = fmadd(R(3), cu, fmul(fmul(R(4.5), cu), cu));
  return fmul(w, fmadd(R(1) + drho, fmadd(R(-1.5), uu, t), drho));
}
// 3 cu + 4.5 cu^2 - usq15 and the shifted equilibrium w (drho + rho b)
__device__ __forceinline__ float heq_of(float w, float drho, float rho, float cu, float usq15) {
  return w * (drho + rho * (3.f * cu + 4.5f * cu * cu - usq15));
}
__device__ __forceinline__ double heq_of(double w, double drho, double rho, double cu, double usq15) {
  return w * fmadd(rho, fmadd(fmadd(4.5, cu, 3.0), cu, -usq15), drho);
}

// Shifted equilibrium of direction i at (drho, rho, u).
template <typename R>
__device__ __forceinline__ R heq(int i, R drho, R rho, R ux, R uy, R uz, R usq15) {
  return heq_of(wgt<R>(i), drho, rho, cdotu<R>(i, ux, uy, uz), usq15);
}

// What the collision of a site takes from its sums drho = sum h and j = sum h c:
// rest(h) is the post-collision population of direction 0, side(c, .., h) of a
// direction of weight class c (1: axis, 2: diagonal) given its pair's c.u or c.j
// and the sign that tells the pair's two directions apart.
template <typename R> struct Bgk;

// FP32.  A pair shares a = 4.5 (c.u)^2 - 1.5 u.u, and its two equilibria are
// w (drho + rho (a +- 3 c.u)); h' = (1 - omega) h + omega heq, with omega w rho
// and omega w drho formed once per weight class, is two fused multiply-adds
// per direction.
template <> struct Bgk<float> {
  float ux, uy, uz, usq15, om1, wr[3], wd[3];  // wr, wd: omega w rho, omega w drho for w = 1/3, 1/18, 1/36
  __device__ __forceinline__ Bgk(float drho, float jx, float jy, float jz, float omega) {
    const float rho = 1.f + drho;
    const float inv = 1.f / rho;
    ux = jx * inv;
    uy = jy * inv;
    uz = jz * inv;
    usq15 = 1.5f * fmadd(uz, uz, fmadd(uy, uy, ux * ux));
    om1 = 1.f - omega;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float ow = omega * wgt<float>(c == 0 ? 0 : (c == 1 ? 1 : 7));
      wr[c] = ow * rho;
      wd[c] = ow * drho;
    }
  }
  __device__ __forceinline__ float rest(float h) const { return fmadd(om1, h, fmadd(-wr[0], usq15, wd[0])); }
  __device__ __forceinline__ float side(int c, float cu, float k, float h) const {
    const float a = fmadd(4.5f * cu, cu, -usq15);
    return fmadd(om1, h, fmadd(c == 1 ? wr[1] : wr[2], fmadd(k, cu, a), c == 1 ? wd[1] : wd[2]));
  }
};

// FP64, which GB300 runs at 1/64 of the FP32 rate: the FP64 step kernels are
// bound by the number of these operations.  With rho u = j a pair's two values
// are (1 - omega) h + e +- b c.j, e = T (c.j)^2 + A, where A = w omega (drho -
// 1.5 j.j / rho), T = 4.5 w omega / rho and b = 3 w omega per weight class: six
// operations a pair after c.j, none of them for u.
template <> struct Bgk<double> {
  double jx, jy, jz, om1, A[3], T[2], B[2];  // T, B: w = 1/18, 1/36
  __device__ __forceinline__ Bgk(double drho, double x, double y, double z, double omega) : jx(x), jy(y), jz(z) {
    const double t = omega * (1.0 / (1.0 + drho));
    const double jj = fmadd(jz, jz, fmadd(jy, jy, jx * jx));
    const double a = fmadd(-1.5 * t, jj, omega * drho);
    om1 = 1.0 - omega;
    A[0] = a * (1.0 / 3.0);
    A[1] = a * (1.0 / 18.0);
    A[2] = 0.5 * A[1];
    T[0] = 0.25 * t;
    T[1] = 0.125 * t;
    B[0] = omega * (1.0 / 6.0);
    B[1] = 0.5 * B[0];
  }
  __device__ __forceinline__ double rest(double h) const { return fmadd(om1, h, A[0]); }
  __device__ __forceinline__ double side(int c, double cj, double sign, double h) const {
    const double e = fmadd((c == 1 ? T[0] : T[1]) * cj, cj, c == 1 ? A[1] : A[2]);
    return fmadd(om1, h, fmadd(sign * (c == 1 ? B[0] : B[1]), cj, e));
  }
};

// c.v of direction i, whose first nonzero component is positive (odd i).
template <typename R>
__device__ __forceinline__ R cdot_pair(int i, R vx, R vy, R vz) {
  if (cx(i)) return cy(i) ? (cy(i) > 0 ? vx + vy : vx - vy) : (cz(i) ? (cz(i) > 0 ? vx + vz : vx - vz) : vx);
  if (cy(i)) return cz(i) ? (cz(i) > 0 ? vy + vz : vy - vz) : vy;
  return vz;
}

// BGK collision (Eq. 3a, dt = 1): h'_i = h_i + omega (heq_i - h_i), handed to
// emit(i, h'_i) direction by direction as each value is final.  Arranged by
// opposite pairs (2p+1, 2p+2), whose c.u differ in sign only: pair sums and
// differences give drho = h_0 + sum (h_2p+1 + h_2p+2) and j = sum (h_2p+1 -
// h_2p+2) c_{2p+1}, and Bgk the rest.  About 140 FP32 instructions a site
// against 210 for the direction-by-direction form, in kernels whose 16-bit
// variants are issue-bound; emitting each pair as soon as it is final lets a
// kernel store it and free its registers.
template <typename R, typename Emit>
__device__ __forceinline__ void collide_emit(const R* h, R omega, Emit&& emit) {
  R drho = h[0], jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const int i = 2 * p + 1;
    const R sp = h[i] + h[i + 1], dp = h[i] - h[i + 1];
    drho += sp;
    if (cx(i)) jx = cx(i) > 0 ? jx + dp : jx - dp;
    if (cy(i)) jy = cy(i) > 0 ? jy + dp : jy - dp;
    if (cz(i)) jz = cz(i) > 0 ? jz + dp : jz - dp;
  }
  const Bgk<R> b(drho, jx, jy, jz, omega);
  emit(0, b.rest(h[0]));
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const int i = 2 * p + 1, c = i <= 6 ? 1 : 2;
    if constexpr (sizeof(R) == 4) {
      const R cu = cdotu<R>(i, b.ux, b.uy, b.uz);
      emit(i, b.side(c, cu, R(3), h[i]));
      emit(i + 1, b.side(c, cu, R(-3), h[i + 1]));
    } else {
      const R cj = cdot_pair<R>(i, b.jx, b.jy, b.jz);
      emit(i, b.side(c, cj, R(1), h[i]));
      emit(i + 1, b.side(c, cj, R(-1), h[i + 1]));
    }
  }
}

// The collision in place.
template <typename R>
__device__ __forceinline__ void collide(R* h, R omega) {
  R out[Q];
  collide_emit<R>(h, omega, [&](int i, R v) { out[i] = v; });
#pragma unroll
  for (int i = 0; i < Q; ++i) h[i] = out[i];
}

// ---------------------------------------------------------------------------
// Gather of the pre-collision state f(t) at site x from the post-collision
// state s'(t-1) (pull streaming, Eq. 3b) with boundaries:
//   fluid source:   h_i = s'_i(x - c_i)
//   wall link:      h_i = s'_ibar(x)                         (bounce-back)
//   velocity iolet: h_i = s'_ibar(x) + coef rho_s A          (Ladd)
//   pressure iolet: h_i = f^eq_i(rho_k, u_g) - w_i           (ghost density)
// rho_s, u_s are the moments of s'(t-1) at x: BGK conserves mass and
// momentum, so they equal the pre-collision moments at time t-1 that the
// paper's push formulation uses for these boundaries.
// ---------------------------------------------------------------------------
// Boundary values of iolet links at site x (rare: only iolet sites).  On
// entry h[i] of an iolet link already holds s'_ibar(x) (the gather selects
// the own opposite slot for every non-fluid source).  All index codes and
// link records are loaded up front, independently of each other, so the
// loads overlap instead of forming a chain per direction.
template <typename S>
__device__ __forceinline__ void iolet_fixup(const S* __restrict__ fin, const int32_t* __restrict__ src,
                                            const LinkRec* __restrict__ links, const double* __restrict__ amp,
                                            const StepParams& p, int64_t x, typename Real<S>::type* h) {
  using R = typename Real<S>::type;
  const int64_t n = p.n;
  int32_t code[Q];
#pragma unroll
  for (int i = 1; i < Q; ++i) code[i] = src[(int64_t)(i - 1) * p.sn + x];
  // moments of the site's own post-collision state s'(t-1)
  R d = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    R v = ldpop(fin + (int64_t)i * n + x);
    d += v;
    if (cx(i)) jx += cx(i) > 0 ? v : -v;
    if (cy(i)) jy += cy(i) > 0 ? v : -v;
    if (cz(i)) jz += cz(i) > 0 ? v : -v;
  }
  const R rho_s = R(1) + d;
  const R ux = jx / rho_s, uy = jy / rho_s, uz = jz / rho_s;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const bool io = code[i] <= -2;
    const LinkRec L = links[io ? -code[i] - 2 : 0];       // record 0 exists whenever a site has an iolet link
    const R a = BC<R>::amp(p, amp, L.kind == 0 && L.group >= 0 ? L.group : 0);
    if (!io) continue;
    const IoletParam& iop = p.io[L.iolet];
    if (L.kind == 0) {
      R rho = p.ladd_rho_one ? R(1) : rho_s;
      h[i] += BC<R>::coef(L) * rho * a * BC<R>::val(p, L.iolet);
    } else {
      R gx = ux, gy = uy, gz = uz;
      if (!p.ghost_full_u) {
        R un = dot3(gx, gy, gz, BC<R>::nx(iop), BC<R>::ny(iop), BC<R>::nz(iop));
        gx = un * BC<R>::nx(iop);
        gy = un * BC<R>::ny(iop);
        gz = un * BC<R>::nz(iop);
      }
      R drho = BC<R>::val(p, L.iolet);
      h[i] = ghost_heq<R>(wgt<R>(i), drho, cdotu<R>(i, gx, gy, gz), dot3(gx, gy, gz, gx, gy, gz));
    }
  }
}

// ---------------------------------------------------------------------------
// Warp-cooperative boundary sites: a lane per direction (the adjoint: one
// warp a site, lanes 19..31 idle; the forward kernels: a half-warp a site,
// three lanes holding two directions).  Moments are summed by a shuffle loop
// in direction order with exactly the operations of the per-thread code
// above, so a site gets bit-identical values whichever path processes it.
// ---------------------------------------------------------------------------
constexpr unsigned FULL_MASK = 0xffffffffu;
static __constant__ int8_t k_cx[32] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
static __constant__ int8_t k_cy[32] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
static __constant__ int8_t k_cz[32] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};

__device__ __forceinline__ int lane_opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
template <typename R>
__device__ __forceinline__ R lane_w(int i) {
  return i == 0 ? R(1) / R(3) : (i <= 6 ? R(1) / R(18) : R(1) / R(36));
}
template <typename R>
__device__ __forceinline__ R lane_cdotu(int i, R ux, R uy, R uz) {
  R s = R(0);
  if (k_cx[i]) s += k_cx[i] > 0 ? ux : -ux;
  if (k_cy[i]) s += k_cy[i] > 0 ? uy : -uy;
  if (k_cz[i]) s += k_cz[i] > 0 ? uz : -uz;
  return s;
}
template <typename R>
__device__ __forceinline__ R lane_heq(int i, R drho, R rho, R ux, R uy, R uz, R usq15) {
  return heq_of(lane_w<R>(i), drho, rho, lane_cdotu<R>(i, ux, uy, uz), usq15);
}
// (sum v, sum v c) over lanes 0..18 in direction order; sgn = -1 sums -v c
template <typename R>
__device__ __forceinline__ void lane_moment_sums(R v, R sgn, R* d, R* jx, R* jy, R* jz) {
  R a = R(0), x = R(0), y = R(0), z = R(0);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const R vk = __shfl_sync(FULL_MASK, v, k);
    a += vk;
    if (cx(k)) x += (cx(k) > 0) == (sgn > R(0)) ? vk : -vk;
    if (cy(k)) y += (cy(k) > 0) == (sgn > R(0)) ? vk : -vk;
    if (cz(k)) z += (cz(k) > 0) == (sgn > R(0)) ? vk : -vk;
  }
  *d = a; *jx = x; *jy = y; *jz = z;
}
// Boundary value of the lane's iolet link (as iolet_fixup computes it):
// `out` = s'_ibar(x); rho_s, u_s the moments of the stored post-collision
// state; val the iolet's boundary value (BC<R>::val).
template <typename R>
__device__ __forceinline__ R lane_iolet_value(int i, const LinkRec& L, R out, R rho_s, R ux, R uy, R uz, R a, R val,
                                              const StepParams& p) {
  const IoletParam& iop = p.io[L.iolet];
  if (L.kind == 0) {
    R rho = p.ladd_rho_one ? R(1) : rho_s;
    return out + BC<R>::coef(L) * rho * a * val;
  }
  R gx = ux, gy = uy, gz = uz;
  if (!p.ghost_full_u) {
    R un = dot3(gx, gy, gz, BC<R>::nx(iop), BC<R>::ny(iop), BC<R>::nz(iop));
    gx = un * BC<R>::nx(iop);
    gy = un * BC<R>::ny(iop);
    gz = un * BC<R>::nz(iop);
  }
  R drho = val;
  return ghost_heq<R>(lane_w<R>(i), drho, lane_cdotu<R>(i, gx, gy, gz), dot3(gx, gy, gz, gx, gy, gz));
}

// ---------------------------------------------------------------------------
// Reading f(t) from a population buffer (read modes of hlb_internal.h:
// 0 = in place, 1 = pull A-B gather with boundaries, 2 = AA gather).
// ---------------------------------------------------------------------------
// Address of slot i of site x in an odd step (and in an AA read-back): the
// population arriving along c_i was written by the source x - c_i into its
// opposite slot, or, for a non-fluid source, by x itself into slot i.
__device__ __forceinline__ int64_t aa_addr(int i, int32_t s, int64_t n, int64_t x) {
  return s >= 0 ? (int64_t)opp(i) * n + s : (int64_t)i * n + x;
}

// ---------------------------------------------------------------------------
// Offsets of the hot kernels.  A thread keeps up to 18 slot offsets in
// registers, so they are 32-bit.  With WIDE = false (19 x the index row
// stride below 2^32, about 226M sites) an offset is the element offset from
// the array base.  With WIDE = true it is the offset within the direction
// pair (2p-1, 2p), p = (i + 1) / 2, whose two rows are contiguous and start
// at element (2p - 1) n: every gather or store of a step touches only
// direction i and opp(i), both in that pair, and offsets there stay below
// 2n < 2^32 for any lattice of fewer than 2^31 sites.  The 64-bit pair start
// is added when the address is formed.
// ---------------------------------------------------------------------------
// offset of row `row` (i or opp(i), i >= 1) at site e
template <bool WIDE>
__device__ __forceinline__ uint32_t slot(int row, uint32_t n, uint32_t e) {
  return WIDE ? ((row & 1) ? e : n + e) : (uint32_t)row * n + e;
}
// address of a slot of direction i's pair
template <bool WIDE, typename T>
__device__ __forceinline__ T* at(T* a, int i, uint32_t n, uint32_t off) {
  return WIDE ? a + ((uint64_t)(2 * ((i + 1) >> 1) - 1) * n + off) : a + off;
}
// index code of direction i >= 1 at site x (rows of stride sn)
template <bool WIDE>
__device__ __forceinline__ const int32_t* idx_at(const int32_t* src, int i, uint32_t sn, uint32_t x) {
  return WIDE ? src + ((uint64_t)(i - 1) * sn + x) : src + (uint32_t)(i - 1) * sn + x;
}

// ---------------------------------------------------------------------------
// Compact index table, one of two forms for each tile of CT_TILE sites.
//
// Row form.  A lattice is ordered lexicographically by (z, y, x), so the
// sites of one lattice row (y, z) are consecutive wherever the row has no
// hole, and the 18 sources x - c_i of a site lie in nine rows: its own, at
// x -+ 1, and eight others, in each of which the sources of the directions
// with the same (cy, cz) are neighbours: s = p - cx with one position p for
// up to three directions.  p - x changes by a few sites from row to row, so
// over a tile it fits 8 bits above the tile's smallest.  Per site three
// 32-bit words (rows of stride sn in rtab): the bit mask of the directions
// with a fluid source (bit i - 1; bit CT_IOLET_BIT: the site has an iolet
// link), and the eight 8-bit offsets, group g in byte g % 4 of word 1 + g / 4.
// Per tile the eight bases (rbase[tile][g], smallest p - x of the group).
// 12.1 bytes a site.
//
// Offset form, for the tiles that a hole in a row or a wide span keeps out
// of the row form (1.9 % of the tiles of the seeded 20M-site tree, 14 % at
// 0.5M sites): per tile and direction the smallest fluid source
// (tbase[tile][i - 1], CT_BASES int32 entries a tile, the last two unused),
// and per site and direction a 16-bit offset from it, or CT_WALL / CT_IOLET
// for a link without a fluid source.  Directions 2p + 1 (low half) and 2p + 2
// (high half) share one 32-bit word in row p of ctab (rows of stride sn): 36
// bytes a site.  rbase[tile][0] = CT_NO_ROWS marks such a tile.
//
// A lattice with a span above CT_MAX_SPAN in some tile uses the 32-bit table
// (72 bytes a site; the same kernels with CT = false).
// ---------------------------------------------------------------------------
constexpr uint32_t CT_WALL = 0xffffu, CT_IOLET = 0xfffeu, CT_MAX_SPAN = 0xfffdu;
constexpr int CT_TILE = 256, CT_BASES = 20;
constexpr int CT_GROUPS = 8, CT_ROW_WORDS = 3, CT_IOLET_BIT = 18;
constexpr int32_t CT_NO_ROWS = (int32_t)0x80000000;

// Row-form group of direction i by (cy, cz); CT_GROUPS for the site's own row.
__host__ __device__ constexpr int row_group(int i) {
  return cz(i) == 0 ? (cy(i) == 0 ? CT_GROUPS : (cy(i) > 0 ? 0 : 1))
                    : (cy(i) == 0 ? (cz(i) > 0 ? 2 : 3)
                                  : (cz(i) > 0 ? (cy(i) > 0 ? 4 : 7) : (cy(i) > 0 ? 6 : 5)));
}

// The streaming index of a lattice as the kernels read it.
struct IndexTables {
  const int32_t* src;     // [18][sn] int32 codes
  const uint32_t* ctab;   // [9][sn] offset form
  const int32_t* tbase;   // [tiles][CT_BASES]
  const uint32_t* rtab;   // [CT_ROW_WORDS][sn] row form
  const int32_t* rbase;   // [tiles][CT_GROUPS]
  const uint32_t* imask;  // [(n + 31) / 32] bit x % 32 of word x / 32: site x has an iolet link
};

// How a kernel loads its index entries: read-only cached, or streaming (read
// once, evict first).
enum { LD_NC = 0, LD_STREAM = 1 };
template <int LD, typename T>
__device__ __forceinline__ T ld_index(const T* p) {
  return LD == LD_STREAM ? __ldcs(p) : __ldg(p);
}

// The offset-form entries of site x: w[9] from ctab, b[i - 1] the tile's bases.
template <bool WIDE, int LD>
__device__ __forceinline__ void load_offset_form(const IndexTables& ix, uint32_t sn, uint32_t x, uint32_t tile,
                                                 uint32_t* w, int32_t* b) {
#pragma unroll
  for (int q = 0; q < 9; ++q)
    w[q] = ld_index<LD>(WIDE ? ix.ctab + ((uint64_t)q * sn + x) : ix.ctab + (uint32_t)q * sn + x);
  const int4* tb = reinterpret_cast<const int4*>(ix.tbase + (uint64_t)tile * CT_BASES);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const int4 v = __ldg(tb + q);
    b[4 * q] = v.x;
    b[4 * q + 1] = v.y;
    b[4 * q + 2] = v.z;
    b[4 * q + 3] = v.w;
  }
}
// 16-bit offset of direction i among the words w[9] of a site.
__device__ __forceinline__ uint32_t offset_of(const uint32_t* w, int i) {
  return (i & 1) ? (w[(i - 1) >> 1] & 0xffffu) : (w[(i - 1) >> 1] >> 16);
}
// The tile's row-form bases; false if the tile has the offset form.
__device__ __forceinline__ bool load_row_bases(const IndexTables& ix, uint32_t tile, int32_t* b) {
  const int4* rb = reinterpret_cast<const int4*>(ix.rbase + (uint64_t)tile * CT_GROUPS);
  const int4 lo = __ldg(rb), hi = __ldg(rb + 1);
  b[0] = lo.x;
  b[1] = lo.y;
  b[2] = lo.z;
  b[3] = lo.w;
  b[4] = hi.x;
  b[5] = hi.y;
  b[6] = hi.z;
  b[7] = hi.w;
  return b[0] != CT_NO_ROWS;
}
// Row positions p of site x's eight groups from its two offset words; pos[8] = x.
__device__ __forceinline__ void row_positions(uint32_t x, const int32_t* b, uint32_t w1, uint32_t w2, uint32_t* pos) {
#pragma unroll
  for (int g = 0; g < CT_GROUPS; ++g) pos[g] = x + (uint32_t)b[g] + (((g < 4 ? w1 : w2) >> (8 * (g & 3))) & 0xffu);
  pos[CT_GROUPS] = x;
}

// Calls link(i, fluid, s) for the 18 directions i of site x: whether the link
// has a fluid source, and if so its index s.  Offset form:
template <bool WIDE, int LD, typename Link>
__device__ __forceinline__ void offset_links(const IndexTables& ix, uint32_t sn, uint32_t x, uint32_t tile, Link&& link) {
  uint32_t w[9];
  int32_t b[CT_BASES];
  load_offset_form<WIDE, LD>(ix, sn, x, tile, w, b);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const uint32_t o = offset_of(w, i);
    link(i, o < CT_IOLET, (uint32_t)b[i - 1] + o);
  }
}
// Whichever form the tile has.  The row form costs three loads of words a site
// and about two integer instructions a direction before the caller's select,
// against nine loads and four instructions for the offset form.  Returns
// whether the site has an iolet link (IOLET: asked for).
template <bool CT, bool WIDE, int LD, bool IOLET, typename Link>
__device__ __forceinline__ bool for_links(const IndexTables& ix, uint32_t sn, uint32_t x, uint32_t tile, Link&& link) {
  if (CT) {
    int32_t b[CT_GROUPS];
    if (load_row_bases(ix, tile, b)) {
      uint32_t w[CT_ROW_WORDS], pos[CT_GROUPS + 1];
#pragma unroll
      for (int q = 0; q < CT_ROW_WORDS; ++q)
        w[q] = ld_index<LD>(WIDE ? ix.rtab + ((uint64_t)q * sn + x) : ix.rtab + (uint32_t)q * sn + x);
      row_positions(x, b, w[1], w[2], pos);
#pragma unroll
      for (int i = 1; i < Q; ++i) link(i, (w[0] >> (i - 1)) & 1u, pos[row_group(i)] - (uint32_t)cx(i));
      return IOLET && ((w[0] >> CT_IOLET_BIT) & 1u);
    }
    offset_links<WIDE, LD>(ix, sn, x, tile, link);
  } else {
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const int32_t s = ld_index<LD>(idx_at<WIDE>(ix.src, i, sn, x));
      link(i, s >= 0, (uint32_t)s);
    }
  }
  return IOLET && ((__ldg(ix.imask + (x >> 5)) >> (x & 31)) & 1u);
}

// The 18 codes of site x: code[i] >= 0 is the fluid source of direction i,
// anything negative a link without one.
template <bool CT, bool WIDE, int LD>
__device__ __forceinline__ void load_codes(const IndexTables& ix, uint32_t sn, uint32_t x, uint32_t tile, int32_t* code) {
  for_links<CT, WIDE, LD, false>(ix, sn, x, tile, [&](int i, bool fluid, uint32_t s) { code[i] = fluid ? (int32_t)s : -1; });
}

// The 18 population offsets a pull step gathers from at site x (off[i], i =
// 1..18): for a fluid source s the slot of row i at s, otherwise row opp(i) at
// x itself, which is bounce-back (iolet links get their values elsewhere).
// Returns whether the site has an iolet link.
template <bool CT, bool WIDE, int LD>
__device__ __forceinline__ bool load_offsets(const IndexTables& ix, uint32_t sn, uint32_t n, uint32_t x, uint32_t tile,
                                             uint32_t* off) {
  return for_links<CT, WIDE, LD, true>(ix, sn, x, tile, [&](int i, bool fluid, uint32_t s) {
    off[i] = fluid ? slot<WIDE>(i, n, s) : slot<WIDE>(opp(i), n, x);
  });
}

// f(t) at site x (tile `tile`), and the bits of the directions with a fluid
// source (bit i - 1) when FLUID or the gather needs them.  The index rows are
// addressed in 64 bits: these kernels read them once a call, not once a step.
template <typename S, int MODE, bool CT, bool FLUID>
__device__ __forceinline__ uint32_t load_state(const S* __restrict__ fin, const IndexTables& ix,
                                               const LinkRec* __restrict__ links, const double* __restrict__ amp,
                                               const StepParams& p, int64_t x, uint32_t tile, typename Real<S>::type* h) {
  const int64_t n = p.n;
  uint32_t fluid = 0;
  h[0] = ldpop(fin + x);
  bool iolet = false;
  if (MODE != 0 || FLUID)
    iolet = for_links<CT, true, LD_NC, MODE == 1>(ix, (uint32_t)p.sn, (uint32_t)x, tile, [&](int i, bool f, uint32_t s) {
      if (FLUID) fluid |= f ? 1u << (i - 1) : 0u;
      if (MODE == 1) h[i] = ldpop(fin + (f ? (int64_t)i * n + s : (int64_t)opp(i) * n + x));
      if (MODE == 2) h[i] = ldpop(fin + (f ? (int64_t)opp(i) * n + s : (int64_t)i * n + x));
    });
  if (MODE == 0) {
#pragma unroll
    for (int i = 1; i < Q; ++i) h[i] = ldpop(fin + (int64_t)i * n + x);
  }
  if (MODE == 1 && iolet) iolet_fixup<S>(fin, ix.src, links, amp, p, x, h);
  return fluid;
}

// ---------------------------------------------------------------------------
// Sum of a thread's populations (19 of each of up to 4 sites) for the FP64 mass
// reductions.  GB300 runs FP64 additions and conversions at 1/64 of the FP32
// rate, and 38 of them a site made the reduction take 2.8 times its memory time.
// FP32 values are therefore summed as an unevaluated triple hi + lo + lo2
// (Knuth's two-sum: the rounding error of every addition is exact in FP32; those
// of hi go to lo, those of lo to lo2), converted once a thread.  With u = 2^-24
// and S the sum of the absolute values, only lo2 is rounded on the way: its m
// terms (m <= 76) are u |lo| <= m u^2 S each, so at most m^3 u^3 S < 2^-53 S is
// lost (one site: 2^-59 S), about one rounding of the m - 1 in a chain of FP64
// additions.  (A pair hi + lo keeps only some 2^-43 of S.)  A sum that leaves
// the FP32 range makes lo2 NaN: it is to be taken again in FP64.
// FP32 snapshot of 8.0M sites (two steps, read-out, mass): 750 us; 753 with pairs,
// 777 with a triple converted for every site.
// ---------------------------------------------------------------------------
// *a + b, rounded, into *a; returns the rounding error.
__device__ __forceinline__ float two_sum(float* a, float b) {
  const float s = __fadd_rn(*a, b), t = __fsub_rn(s, *a);
  const float e = __fadd_rn(__fsub_rn(*a, __fsub_rn(s, t)), __fsub_rn(b, t));
  *a = s;
  return e;
}
template <typename R> struct MassSum;
template <> struct MassSum<double> {
  double d = 0;
  __device__ __forceinline__ void add(const double* h) {
#pragma unroll
    for (int i = 0; i < Q; ++i) d += h[i];
  }
  __device__ __forceinline__ bool holds() const { return true; }
  __device__ __forceinline__ double value() const { return d; }
};
template <> struct MassSum<float> {
  float hi = 0.f, lo = 0.f, lo2 = 0.f;
  __device__ __forceinline__ void add(const float* h) {
#pragma unroll
    for (int i = 0; i < Q; ++i) lo2 = __fadd_rn(lo2, two_sum(&lo, two_sum(&hi, h[i])));
  }
  __device__ __forceinline__ bool holds() const { return isfinite(lo2); }
  __device__ __forceinline__ double value() const { return (double)hi + ((double)lo + (double)lo2); }
};
// The sum over `count` sites, load(k, h) giving the k-th.
template <typename R, typename Load>
__device__ __forceinline__ double mass_sum(int count, Load&& load) {
  MassSum<R> m;
  double d = 0;
#pragma unroll 1
  for (bool wide = false;; wide = true) {
#pragma unroll 1
    for (int k = 0; k < count; ++k) {
      R h[Q];
      load(k, h);
      if (wide) {
#pragma unroll
        for (int i = 0; i < Q; ++i) d += (double)h[i];
      } else {
        m.add(h);
      }
    }
    if (wide) return d;
    if (m.holds()) return m.value();
  }
}

// The Windkessel model of an outlet one step on, q its outflow in that step:
// advances rho_c and returns the next ghost density less 1.
__device__ __forceinline__ double wk_advance(double Rp, double C, double Rd, double rho_d, double q, double* rho_c) {
  if (!(C > 0)) return fmadd(Rp + Rd, q, rho_d) - 1.0;
  *rho_c += (q - (*rho_c - rho_d) / Rd) / C;
  return fmadd(Rp, q, *rho_c) - 1.0;
}
// In the pull scheme an outlet's link masses are summed by this many lanes, lane l
// its links l, l + kWkLanes, .. in order, then the lanes of a warp, then the warps.
constexpr int kWkLanes = 64;

// Sites a thread of a mass reduction over a lattice of n takes (a block: that
// many x 256): four, so that the FP64 block sum is paid once for them, but one
// below a million sites, where four sites in a chain take longer than they
// save (43,700 sites: 18.7 us at four).
__host__ __device__ constexpr int mass_sites(int64_t n) { return n < (1 << 20) ? 1 : 4; }

// Post-collision population of a lane's direction i (collide_emit's operations).
template <typename R>
__device__ __forceinline__ R iolet_lane_out(int i, R h, const Bgk<R>& b) {
  if (i == 0) return b.rest(h);
  const int ip = 2 * ((i - 1) >> 1) + 1, c = ip <= 6 ? 1 : 2;
  if constexpr (sizeof(R) == 4)
    return b.side(c, lane_cdotu<R>(ip, b.ux, b.uy, b.uz), (i & 1) ? R(3) : R(-3), h);
  else
    return b.side(c, lane_cdotu<R>(ip, b.jx, b.jy, b.jz), (i & 1) ? R(1) : R(-1), h);
}
// Lanes a site for the iolet sites of the pull step: a site's 19 directions
// spread over them, up to ceil(19 / lanes) a lane (measured on the 20M-site
// tree: BF16 step 418 us at 32, 411 at 16, 405 at 8).
constexpr int kStepIoletLanes = 8;

}  // namespace hlb
