// hlb_multi.cu — many pull A-B steps of a small lattice in one launch.
//
// A lattice of some ten thousand sites steps in about as long as a launch
// takes: 3.4 us for 12k sites, of which the memory and arithmetic are a small
// part.  Here one cooperative launch runs a whole sequence of steps (arXiv
// 2202.11770, Section 3.1 steps 2-5): a thread keeps its site for the launch,
// the gather offsets in registers, and the populations pass from site to site
// through L2 as 64-bit words that hold a value and the number of the step that
// produced it (FP64: two words, half a value each).  A reader polls the word
// itself, so a step costs one trip to L2 and back: no barrier, no fence, no
// flag.  A grid of flags with a release and an acquire a step measured 3.8 us
// a step at 12k sites, slower than the launches (this form: 2.4).
//
// Two word buffers, by step parity.  A site overwrites the words of step k - 1
// at step k + 1, after it has read step k of every site it pulls from; those
// had read its words of step k - 1 before they produced step k.  This needs
// every link to be mutual (y pulls from x when x pulls from y), which create
// checks; other lattices are stepped launch by launch.
//
// Sites with iolet links are stepped by blocks of their own,
// kStepIoletLanes lanes a site, with links and codes in registers; a
// Windkessel outlet has a block that sums the outlet's link masses and
// hands the next ghost density back, both through words of the same kind.
//
// Every wait is bounded.  The cooperative launch makes all blocks resident, so
// no wait runs out in a correct run.  A thread whose wait does run out sets the
// solver's status word, which the next synchronising call returns as
// HLB_ERR_WAIT, leaves NaN in what it would have written (its site's
// populations, its outlet's model) and returns.
#include <algorithm>

#include "hlb_internal.h"

using namespace hlb;

namespace {

constexpr int TB = 64;                     // threads a block
// A thread whose words have not all come sleeps this long before it asks again:
// the polls of the others load L2 less (50k sites 4.1 -> 3.8 us a step).
constexpr unsigned kPollSleep = 100;  // ns

// Boundary values of the launch's steps, [step][iolet] (BC<R>::val of each).
template <typename R>
struct WaveTable {
  R v[kMultiVals];
};

struct MultiArgs {
  IndexTables ix;
  const LinkRec* links;
  const double* amp;
  const int32_t* sites;   // iolet sites, ascending
  int64_t nsites;
  uint64_t* word;         // [2][18][n] words (FP64: [2][18][n][2])
  uint64_t* flux;         // [links][2] link masses, FP64 words
  uint64_t* ghost;        // [iolets][2] ghost densities less 1, FP64 words
  uint32_t tag0;          // number of the launch's first step
  uint32_t limit[kMultiWaits];  // polls after which a wait of each kind (WAIT_BULK ..) gives up
  uint32_t* status;       // set to 1 by a wait that ran out
  int32_t nbulk, niolet, nsteps;
  // Windkessel outlets
  const int64_t* begin;   // link ranges per iolet
  const double* wkpar;
  double* wkstate;
  double* iovnext;
};

__device__ __forceinline__ uint64_t ld_word(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t pack(uint32_t v, uint32_t tag) { return ((uint64_t)tag << 32) | v; }

// A value with its step number: one word for FP32 and 16-bit storage (the
// stored value as FP32), two for FP64.
template <typename R> struct Word;
template <> struct Word<float> {
  static constexpr int N = 1;
  uint64_t w;
  __device__ __forceinline__ void load(const uint64_t* p) { w = ld_word(p); }
  __device__ __forceinline__ bool is(uint32_t tag) const { return (uint32_t)(w >> 32) == tag; }
  __device__ __forceinline__ float value() const { return __uint_as_float((uint32_t)w); }
  static __device__ __forceinline__ void store(uint64_t* p, float v, uint32_t tag) { st_word(p, pack(__float_as_uint(v), tag)); }
};
template <> struct Word<double> {
  static constexpr int N = 2;
  uint64_t w, z;
  __device__ __forceinline__ void load(const uint64_t* p) {
    w = ld_word(p);
    z = ld_word(p + 1);
  }
  __device__ __forceinline__ bool is(uint32_t tag) const { return (uint32_t)(w >> 32) == tag && (uint32_t)(z >> 32) == tag; }
  __device__ __forceinline__ double value() const { return __hiloint2double((int)(uint32_t)z, (int)(uint32_t)w); }
  static __device__ __forceinline__ void store(uint64_t* p, double v, uint32_t tag) {
    st_word(p, pack((uint32_t)__double2loint(v), tag));
    st_word(p + 1, pack((uint32_t)__double2hiint(v), tag));
  }
};
// One value, waited for; *late set when the wait runs out.  Its limit is a
// constant: with one from the launch's arguments the same loop left the lanes
// of an iolet warp apart, and a step with outlet models took 8.9 us instead of
// 7.7 (50k sites); other forms of the loop cost more.
constexpr unsigned kGhostPolls = 1u << 20;
__device__ __forceinline__ double wait_double(const uint64_t* p, uint32_t tag, bool* late) {
  Word<double> v;
  unsigned spins = 0;
  for (v.load(p); !v.is(tag); v.load(p))
    if (++spins > kGhostPolls) {
      *late = true;
      break;
    }
  return v.value();
}
// The value as it is stored.
template <typename S>
__device__ __forceinline__ typename Real<S>::type rounded(typename Real<S>::type v) {
  return to_real(from_real<S>(v));
}
template <typename S>
__device__ __forceinline__ S not_a_number() {
  return from_real<S>(typename Real<S>::type(__int_as_float(0x7fc00000)));
}
__device__ __forceinline__ void ran_out(const MultiArgs& a) { *(volatile uint32_t*)a.status = 1u; }

template <typename S>
__device__ __forceinline__ void bulk_block(const S* in, S* out, const MultiArgs& a, const StepParams& p, int b) {
  using R = typename Real<S>::type;
  using W = Word<R>;
  const uint32_t n = (uint32_t)p.n, x = (uint32_t)(b * TB) + threadIdx.x;
  if (x >= n) return;
  uint32_t off[Q];
  if (load_offsets<true, false, LD_NC>(a.ix, (uint32_t)p.sn, n, x, x / CT_TILE, off)) return;  // an iolet site
  const R omega = omega_of<R>(p);
  R h[Q];
  h[0] = to_real(in[x]);
#pragma unroll
  for (int i = 1; i < Q; ++i) h[i] = to_real(in[off[i]]);
  for (int k = 0;; ++k) {
    const bool last = k == a.nsteps - 1;
    uint64_t* put = a.word + (int64_t)(k & 1) * (Q - 1) * n * W::N;
    const uint32_t tag = a.tag0 + (uint32_t)k;
    R rest = R(0);
    collide_emit<R>(h, omega, [&](int i, R v) {
      v = rounded<S>(v);
      if (i == 0)
        rest = v;
      else if (!last)
        W::store(put + (uint64_t)((uint32_t)(i - 1) * n + x) * W::N, v, tag);
      if (last) out[(uint32_t)i * n + x] = from_real<S>(v);
    });
    if (last) return;
    W w[Q];
    unsigned spins = 0;
    while (true) {
      bool all = true;
#pragma unroll
      for (int i = 1; i < Q; ++i) w[i].load(put + (uint64_t)(off[i] - n) * W::N);
#pragma unroll
      for (int i = 1; i < Q; ++i) all &= w[i].is(tag);
      if (all) break;
      if (sizeof(S) < 8) __nanosleep(kPollSleep);  // FP64: 11.6 us a step without, 17.7 with
      if (++spins > a.limit[WAIT_BULK]) {
#pragma unroll 1
        for (int i = 0; i < Q; ++i) out[(uint32_t)i * n + x] = not_a_number<S>();
        ran_out(a);
        return;
      }
    }
    h[0] = rest;
#pragma unroll
    for (int i = 1; i < Q; ++i) h[i] = w[i].value();
  }
}

// The boundary-value arithmetic of step_iolet_site (hlb_forward.cu), with the
// site's codes, link records and amplitudes held over the steps.
template <typename S>
__device__ __forceinline__ void iolet_block(const S* in, S* out, const MultiArgs& a,
                                            const WaveTable<typename Real<S>::type>& wave, const StepParams& p, int j) {
  using R = typename Real<S>::type;
  using WD = Word<R>;
  constexpr int W = kStepIoletLanes, NE = (Q + W - 1) / W;
  const int64_t site = ((int64_t)j * TB + threadIdx.x) / W;
  const bool live = site < a.nsites;  // lanes past the end compute along and touch nothing
  const int hl = threadIdx.x & (W - 1), K = p.n_iolets;
  const uint32_t n = (uint32_t)p.n, x = (uint32_t)a.sites[live ? site : 0];
  int32_t c[NE];
  uint32_t from[NE];  // slot that the lane's direction is gathered from
  int io[NE], kind[NE];
  R amp[NE], coef[NE], h[NE], own[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    c[e] = (i >= 1 && i < Q) ? a.ix.src[(int64_t)(i - 1) * p.sn + x] : 0;
    from[e] = i == 0 ? x : (i < Q ? (c[e] >= 0 ? (uint32_t)i * n + (uint32_t)c[e] : (uint32_t)lane_opp(i) * n + x) : x);
    const LinkRec L = a.links[c[e] <= -2 ? -c[e] - 2 : 0];
    io[e] = L.iolet;
    kind[e] = L.kind;
    coef[e] = BC<R>::coef(L);
    amp[e] = BC<R>::amp(p, a.amp, L.kind == 0 && L.group >= 0 ? L.group : 0);
    h[e] = i < Q ? to_real(in[from[e]]) : R(0);
    own[e] = i < Q ? to_real(in[(uint32_t)i * n + x]) : R(0);
  }
  const R omega = omega_of<R>(p);
  // A wait of some lane of the warp ran out: the warp's sites end here.
  auto give_up = [&](bool late) {
    if (!__any_sync(FULL_MASK, late)) return false;
#pragma unroll 1
    for (int i = hl; live && i < Q; i += W) out[(uint32_t)i * n + x] = not_a_number<S>();
    if (late) ran_out(a);
    return true;
  };
  for (int k = 0;; ++k) {
    const bool last = k == a.nsteps - 1;
    uint64_t* put = a.word + (int64_t)(k & 1) * (Q - 1) * n * WD::N;
    const uint32_t tag = a.tag0 + (uint32_t)k;
    bool late = false;
    // moments of the site's own post-collision state, then the boundary values
    R d = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const R vk = __shfl_sync(FULL_MASK, own[q / W], q % W, W);
      d += vk;
      if (cx(q)) jx += cx(q) > 0 ? vk : -vk;
      if (cy(q)) jy += cy(q) > 0 ? vk : -vk;
      if (cz(q)) jz += cz(q) > 0 ? vk : -vk;
    }
    const R rho_s = R(1) + d;
    const R ux = jx / rho_s, uy = jy / rho_s, uz = jz / rho_s;
#pragma unroll
    for (int e = 0; e < NE; ++e)
      if (c[e] <= -2) {
        R val = wave.v[k * K + io[e]];
        const bool coupled = (p.coupled[io[e] >> 6] >> (io[e] & 63)) & 1ull;
        // the outlet's block sends the ghost density of step k >= 2 with that step's number
        if (coupled && live) val = R(k == 0 ? p.ioval[io[e]] : (k == 1 ? a.iovnext[io[e]] : wait_double(a.ghost + 2 * io[e], tag, &late)));
        const R o = h[e];
        LinkRec L;
        L.kind = (int8_t)kind[e];
        L.iolet = (int16_t)io[e];
        L.coef = coef[e];
        L.coef_f = (float)coef[e];
        h[e] = lane_iolet_value<R>(e * W + hl, L, o, rho_s, ux, uy, uz, amp[e], val, p);
        if (coupled && live && k > 0) {
          // the outflow as k_wk_update takes it, its velocity by the reciprocal
          const R inv = R(1) / rho_s;
          const R m = lane_iolet_value<R>(e * W + hl, L, o, rho_s, jx * inv, jy * inv, jz * inv, amp[e], val, p);
          Word<double>::store(a.flux + 2 * (int64_t)(-c[e] - 2), (double)m - (double)o, tag);
        }
      }
    if (give_up(late)) return;
    R drho = __shfl_sync(FULL_MASK, h[0], 0, W), cjx = R(0), cjy = R(0), cjz = R(0);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const int ip = 2 * q + 1;
      const R va = __shfl_sync(FULL_MASK, h[ip / W], ip % W, W), vb = __shfl_sync(FULL_MASK, h[(ip + 1) / W], (ip + 1) % W, W);
      const R sp = va + vb, dp = va - vb;
      drho += sp;
      if (cx(ip)) cjx = cx(ip) > 0 ? cjx + dp : cjx - dp;
      if (cy(ip)) cjy = cy(ip) > 0 ? cjy + dp : cjy - dp;
      if (cz(ip)) cjz = cz(ip) > 0 ? cjz + dp : cjz - dp;
    }
    const Bgk<R> bgk(drho, cjx, cjy, cjz, omega);
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const int i = e * W + hl;
      if (i >= Q) continue;
      own[e] = rounded<S>(iolet_lane_out<R>(i, h[e], bgk));
      if (!live) continue;
      if (i > 0 && !last) WD::store(put + (uint64_t)((uint32_t)(i - 1) * n + x) * WD::N, own[e], tag);
      if (last) out[(uint32_t)i * n + x] = from_real<S>(own[e]);
    }
    if (last) return;
    // what the site gathers next
    WD w[NE];
    unsigned spins = 0;
    while (true) {
      bool all = true;
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const int i = e * W + hl;
        if (live && i >= 1 && i < Q) {  // a lane without a site does not hold writers back: it must not poll
          w[e].load(put + (uint64_t)(from[e] - n) * WD::N);
          all &= w[e].is(tag);
        }
      }
      if (all) break;
      if (++spins > a.limit[WAIT_IOLET]) {
        late = true;
        break;
      }
    }
    if (give_up(late)) return;
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const int i = e * W + hl;
      h[e] = i == 0 ? own[e] : (live && i < Q ? w[e].value() : R(0));
    }
  }
}

// The model of Windkessel outlet number j among the coupled ones, as
// k_wk_update (hlb_forward.cu) advances it, its link masses summed in the same
// order, so that a run gives the same bits however it is cut into launches.  The gather of step k >= 1 applies
// the boundary values of the state that step k - 1 produced, so its link
// masses are that state's outflow; they set the ghost density of step k + 1.
// (The outflow after the last step is k_wk_update's, after this launch.)
__device__ __forceinline__ void wk_block(const MultiArgs& a, const StepParams& p, int j) {
  static_assert(TB == kWkLanes, "the order of the sum");
  __shared__ double sh[TB / 32];
  const int K = p.n_iolets;
  int io = -1;
  for (int k = 0, seen = 0; k < K; ++k)
    if ((p.coupled[k >> 6] >> (k & 63)) & 1ull)
      if (seen++ == j) io = k;
  const double Rp = a.wkpar[4 * io], C = a.wkpar[4 * io + 1], Rd = a.wkpar[4 * io + 2], rho_d = a.wkpar[4 * io + 3];
  double rho_c = a.wkstate[2 * io];
  const int64_t lo = a.begin[io], hi = a.begin[io + 1];
  for (int k = 1; k < a.nsteps; ++k) {
    const uint32_t tag = a.tag0 + (uint32_t)k;
    bool late = false;
    double acc = 0;
    for (int64_t r = lo + threadIdx.x; r < hi && !late; r += TB * 8) {
      Word<double> v[8];
      unsigned spins = 0;
      while (!late) {
        bool all = true;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (r + u * TB < hi) v[u].load(a.flux + 2 * (r + u * TB));
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (r + u * TB < hi) all &= v[u].is(tag);
        if (all) break;
        late = ++spins > a.limit[WAIT_FLUX];
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (r + u * TB < hi) acc += v[u].value();
    }
    if (__syncthreads_or(late)) {
      if (late) ran_out(a);
      if (threadIdx.x == 0) a.wkstate[2 * io] = a.wkstate[2 * io + 1] = a.iovnext[io] = __longlong_as_double(0x7ff8000000000000ll);
      return;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(FULL_MASK, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double flux = 0;
      for (int w = 0; w < TB / 32; ++w) flux += sh[w];
      const double q = -flux;
      const double ghost = wk_advance(Rp, C, Rd, rho_d, q, &rho_c);
      if (k == a.nsteps - 1) {
        a.wkstate[2 * io] = rho_c;
        a.wkstate[2 * io + 1] = q;
        a.iovnext[io] = ghost;
      } else {
        Word<double>::store(a.ghost + 2 * io, ghost, tag + 1u);
      }
    }
  }
}

// Registers: 18 offsets, 18 words in flight and the collision: 96 (FP64 up to 255).
template <typename S> constexpr int multi_per_sm() { return sizeof(S) == 8 ? 4 : 10; }
template <typename S>
__global__ void __launch_bounds__(TB, multi_per_sm<S>()) k_multi(const S* in, S* out, const MultiArgs a,
                                                                 const WaveTable<typename Real<S>::type> wave,
                                                                 const StepParams p) {
  const int b = blockIdx.x;
  // the iolet blocks first: they take longest, and every neighbour waits for them
  if (b < a.niolet)
    iolet_block<S>(in, out, a, wave, p, b);
  else if (b < a.niolet + a.nbulk)
    bulk_block<S>(in, out, a, p, b - a.niolet);
  else
    wk_block(a, p, b - a.niolet - a.nbulk);
}

inline int bulk_blocks(int64_t n) { return (int)((n + TB - 1) / TB); }
inline int iolet_blocks(int64_t nis) { return (int)((nis * kStepIoletLanes + TB - 1) / TB); }
inline int wk_blocks(const hlb_solver* h) {
  int k = 0;
  for (int v : h->wk_on) k += v ? 1 : 0;
  return k;
}

template <typename S>
int resident_blocks(int n_sm) {
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_multi<S>, TB, 0) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per * n_sm;
}

template <typename S>
cudaError_t launch(hlb_solver* h, const void* in, void* out, int64_t t, int m, cudaStream_t s) {
  using R = typename Real<S>::type;
  if (h->multi_tag > UINT32_MAX - (uint32_t)m) {
    // the step numbers start again: clear the words first, so that none left from 2^32
    // steps ago, or never written, is taken for a new one
    const cudaError_t e = cudaMemsetAsync(h->d_word, 0, sizeof(uint64_t) * hlb_multi_words(h->n, h->n_links, h->n_iolets, h->precision), s);
    if (e != cudaSuccess) return e;
    h->multi_tag = 1;
  }
  const StepParams p = h->params(t);
  WaveTable<R> wave;
  const int K = h->n_iolets;
  for (int k = 0; k < m; ++k)
    for (int i = 0; i < K; ++i) {
      const double v = h->wave[i].at((double)(t - 1 + k));
      wave.v[k * K + i] = (R)(h->iolets[i].kind == HLB_VELOCITY ? v : v - 1.0);
    }
  MultiArgs a;
  a.ix = h->index();
  a.links = h->d_links;
  a.amp = h->d_amp;
  a.sites = h->d_iolet_sites;
  a.nsites = h->n_iolet_sites;
  a.word = h->d_word;
  a.flux = h->d_word + 2 * (Q - 1) * h->n * Word<R>::N;
  a.ghost = a.flux + 2 * h->n_links;
  a.tag0 = h->multi_tag;
  for (int k = 0; k < kMultiWaits; ++k) a.limit[k] = h->multi_limit[k];
  a.status = h->d_status;
  a.nbulk = bulk_blocks(h->n);
  a.niolet = iolet_blocks(h->n_iolet_sites);
  a.nsteps = m;
  a.begin = (const int64_t*)(h->d_red + hlb_reduce_partials(h->n));
  a.wkpar = h->d_wkpar;
  a.wkstate = h->d_wkstate;
  a.iovnext = h->d_iovnext;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.nbulk + a.niolet + wk_blocks(h)));
  cfg.blockDim = dim3(TB);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_multi<S>, (const S*)in, (S*)out, (const MultiArgs)a,
                                           (const WaveTable<R>)wave, p);
  // no step number is used twice without the words being cleared in between, so no word of an
  // earlier launch is taken for a new one
  if (e == cudaSuccess) {
    h->multi_tag += (uint32_t)m;
    h->multi_ran = true;
  }
  return e;
}

}  // namespace

size_t hlb_multi_words(int64_t n, int64_t n_links, int32_t n_iolets, int32_t precision) {
  const size_t per = precision == HLB_FP64 ? 2 : 1;
  return 2 * (size_t)(Q - 1) * (size_t)n * per + 2 * (size_t)n_links + 2 * (size_t)n_iolets;
}

int hlb_multi_blocks(const hlb_solver* h) {
  int coop = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device) != cudaSuccess || !coop) {
    cudaGetLastError();
    return 0;
  }
  switch (h->precision) {
    case HLB_FP32: return resident_blocks<float>(h->n_sm);
    case HLB_BF16: return resident_blocks<__nv_bfloat16>(h->n_sm);
    case HLB_FP16: return resident_blocks<__half>(h->n_sm);
    default: return resident_blocks<double>(h->n_sm);
  }
}

// The pull scheme on the compact table with mutual links, all blocks resident,
// enough steps, and outside a stream capture (where the step-by-step launches
// were and stay what is captured).  FP32 and 16 bits up to kMultiSites, where the
// two forms are about to cross: 2.4 us a step against 3.2-3.4 at 12k sites, 2.7 /
// 3.3 at 18k, 3.1 / 3.35 at 24k; at 50k 3.8 / 3.6 (18 words of 8 bytes a site go
// through L2).  FP64 runs at the rate of its arithmetic, spread over more SMs by
// the smaller blocks, 10.2 against 19.8 us at 12k and 14.1 / 19.3 at 24k, so
// whatever fits (about 36k sites).  With Windkessel outlets a step is two
// launches, the second a chain of loads, 7.8 against 10.6 us at 50k, so whatever
// fits as well.
int hlb_multi_steps(const hlb_solver* h, int64_t left) {
  if (h->multi_blocks == 0 || !h->compact || !h->off32 || left < kMultiMin) return 0;
  if (h->n > kMultiSites && h->precision != HLB_FP64 && !h->any_wk()) return 0;
  if (bulk_blocks(h->n) + iolet_blocks(h->n_iolet_sites) + wk_blocks(h) > h->multi_blocks) return 0;
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(h->stream, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return 0;
  }
  const int64_t most = h->n_iolets > 0 ? kMultiVals / h->n_iolets : kMultiVals;
  return (int)std::min(left, most);
}

int hlb_check_waits(hlb_solver* h) {
  if (!h->multi_ran) return HLB_OK;
  uint32_t late = 0;
  cudaError_t e = cudaMemcpyAsync(&late, h->d_status, sizeof late, cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return hlb_cuda_fail(e, "status of a multi-step launch");
  return hlb_wait_status(h, late);
}

int hlb_wait_status(hlb_solver* h, uint32_t late) {
  if (late) return hlb_fail(HLB_ERR_WAIT, "a wait inside a multi-step launch ran out: the state is not valid");
  h->multi_ran = false;
  return HLB_OK;
}

cudaError_t hlb_clear_waits(hlb_solver* h) {
  if (!h->multi_ran) return cudaSuccess;
  h->multi_ran = false;
  return cudaMemsetAsync(h->d_status, 0, sizeof(double), h->stream);
}

extern "C" int hlb_multi_test(hlb_solver* h, const uint32_t* limits, uint32_t next_step, int blocks) {
  if (!h || !limits) return hlb_fail(HLB_ERR_ARG, "null argument");
  for (int k = 0; k < kMultiWaits; ++k) h->multi_limit[k] = limits[k];
  if (next_step) h->multi_tag = next_step;
  if (blocks && h->d_word) h->multi_blocks = blocks;
  return HLB_OK;
}

cudaError_t hlb_launch_multi(hlb_solver* h, const void* in, void* out, int64_t t, int m, cudaStream_t s) {
  switch (h->precision) {
    case HLB_FP32: return launch<float>(h, in, out, t, m, s);
    case HLB_BF16: return launch<__nv_bfloat16>(h, in, out, t, m, s);
    case HLB_FP16: return launch<__half>(h, in, out, t, m, s);
    default: return launch<double>(h, in, out, t, m, s);
  }
}
