// hlb_forward.cu — forward kernels of the D3Q19 sparse-lattice solver.
//
// The step (arXiv 2202.11770, Section 3.2.2: load f, compute rho and u
// (Eqs. 5-6), f^eq (Eq. 4), collide (Eq. 3a), stream (Eq. 3b) with wall and
// iolet boundaries, store) runs as one fused kernel per time step over the
// whole site list; the paper's six per-site-type kernels become one kernel in
// which wall links are branch-free address selects and iolet links a rare
// per-site fix-up.  Two streaming schemes:
//
//  * pull A-B (k_step, k_step2): read buffer A by gathering through the index
//    table, write buffer B; 164 B per FP32 site update with the row form of
//    the compact index table (224 B with the int32 one).
//  * AA pattern (k_aa_even / k_aa_odd and their two-site forms): one
//    buffer.  Even steps read a site's 19 slots and write them back swapped
//    (no index table); odd steps read 19 slots through the index table and
//    write the results to the very same 19 slots.  152 B (even) + 164 B
//    (odd; 224 B with the int32 table) per FP32 update.
//
// The bulk and read-back kernels take the index from its compact form
// (hlb_common.cuh, built by k_ctab_build) unless the lattice does not fit it;
// iolet-site paths, and what reads single sites, use the int32 table.
//
// Read modes of the readback kernels: LOCAL (the buffer holds f(t) in place),
// GATHER_AB (the buffer holds s'(t-1); boundaries applied while gathering),
// GATHER_AA (AA buffer after an even step; boundaries already written).
//
// k_macros: the property cache of Section 3.2.2 step 7 (rho, u) plus WSS.
// k_sums / k_sums_finish: FP64 mass, iolet fluxes and monitor in a fixed order.
#include <math.h>

#include "hlb_internal.h"

using namespace hlb;

namespace {

constexpr int BLOCK = 256;
// Two-site step kernels: threads a block (one tile), and blocks per SM.  Measured
// on the 20M-site tree: 256 threads x 3 blocks ran the BF16 odd step in 415 us,
// 128 x 6 in 394 (a block's slots return sooner), 128 x 7 (72 registers, a few
// bytes of spill) in 388; FP32 532 us at 6 blocks, 539 at 7.
constexpr int PAIR = CT_TILE / 2;
template <typename S> constexpr int pair_blocks() { return sizeof(S) == 4 ? 6 : 7; }

// Lanes a site in the AA iolet pass (8 lanes 1-2 us slower a step on the
// 20M-site tree, 32 lanes 3 us slower).
constexpr int kFixLanes = 16;
constexpr uint32_t kNoTile = 0xffffffffu;  // first tile of a launch without tiles
constexpr int READ = 128;  // threads a block of the read-back kernels, one site each

inline unsigned grid_for(int64_t n) { return (unsigned)((n + BLOCK - 1) / BLOCK); }
inline int64_t mass_blocks(int64_t sites, int per) { return (sites + per * BLOCK - 1) / (per * BLOCK); }

// L2 prefetch hint: `bytes` (a multiple of 16) from a 16-byte aligned address.
__device__ __forceinline__ void l2_prefetch(const void* q, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(q)), "r"(bytes)
               : "memory");
}

// Called by the first warp of a bulk block: prefetch into L2 what the block
// that takes tile `tile` (about a wave of resident blocks later) reads
// first, so that its loads find L2 instead of waiting on DRAM.  Lanes 0-2:
// the tile's row-form index words (256 sites of each).  With POPS, lanes
// 9-26: for direction i = lane - 8, the population row its gathers read
// (ROWOPP: row opp(i), as the AA odd step reads; else row i) from the
// tile's smallest source for i, 320 sites wide (the sources of a tile span
// about 255 sites on vessel lattices).  A tile in the form that is rare in its
// lattice is left to its own loads: where most tiles have the offset form, the
// index words are its nine rows (lanes 0-8) and the bases its own (kPrefetchOffsets
// in `pf`; OFFSETS: asked at all, which the small-lattice form of k_step2 is not:
// the longer code made some of its steps 3 to 10 % slower).  Every range is
// clamped to its array: rtab holds CT_ROW_WORDS rows of sn words, ctab nine, A 19
// rows of n populations.
constexpr uint32_t kPrefetchOffsets = 0x80000000u;
template <typename S, bool POPS, bool ROWOPP, bool OFFSETS>
__device__ __forceinline__ void prefetch_tile(const S* A, const IndexTables& ix, uint32_t n, uint32_t sn,
                                              uint32_t tile, uint32_t pf) {
  const bool offsets = OFFSETS && (pf & kPrefetchOffsets);
  tile += pf & ~kPrefetchOffsets;
  const uint32_t ntiles = (n + BLOCK - 1) / BLOCK;
  const int l = threadIdx.x & 31;
  if (tile >= ntiles) return;
  const uint64_t x0 = (uint64_t)tile * BLOCK;
  if (l < (offsets ? (Q - 1) / 2 : CT_ROW_WORDS)) {
    const uint64_t e = x0 + BLOCK < (uint64_t)sn ? x0 + BLOCK : (uint64_t)sn;  // sn: a multiple of 4
    l2_prefetch((offsets ? ix.ctab : ix.rtab) + (uint64_t)l * sn + x0, (uint32_t)((e - x0) * 4));
  } else if (POPS && l >= 9 && l < 9 + Q - 1) {
    const int i = l - 8, y = k_cy[i], z = k_cz[i];
    const int32_t* rb = ix.rbase + (uint64_t)tile * CT_GROUPS;
    if ((__ldg(rb) == CT_NO_ROWS) != offsets) return;
    // row_group(i) of a run-time direction
    const int g = z == 0 ? (y > 0 ? 0 : 1) : (y == 0 ? (z > 0 ? 2 : 3) : (z > 0 ? (y > 0 ? 4 : 7) : (y > 0 ? 6 : 5)));
    const int64_t first = offsets ? __ldg(ix.tbase + (uint64_t)tile * CT_BASES + (i - 1))
                                  : (int64_t)x0 - k_cx[i] + ((y | z) ? __ldg(rb + g) : 0);
    const uint64_t b = first > 0 ? (uint64_t)first : 0;
    const uint64_t r = ROWOPP ? (uint64_t)lane_opp(i) : (uint64_t)i;
    const uint64_t e = b + 320 < (uint64_t)n ? b + 320 : (uint64_t)n;
    const uint64_t total = ((uint64_t)Q * n * sizeof(S) + 15) & ~15ull;  // within the 256-aligned section
    const uint64_t lo = ((r * n + b) * sizeof(S)) & ~15ull;
    const uint64_t hr = ((r * n + e) * sizeof(S) + 15) & ~15ull;
    const uint64_t hi = hr < total ? hr : total;
    if (b < (uint64_t)n && hi > lo) l2_prefetch(reinterpret_cast<const char*>(A) + lo, (uint32_t)(hi - lo));
  }
}

// ---------------------------------------------------------------------------
// Pull A-B step from f(t) held in place (the first step after initialisation
// or set_state): no gather.
// ---------------------------------------------------------------------------
template <typename S>
__global__ void __launch_bounds__(BLOCK) k_step_local(const S* __restrict__ fin, S* __restrict__ fout,
                                                      const StepParams p) {
  using R = typename Real<S>::type;
  const int64_t n = p.n;
  const int64_t x = (int64_t)blockIdx.x * BLOCK + threadIdx.x;
  pdl_wait();
  pdl_trigger();
  if (x >= n) return;
  R h[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) h[i] = ldpop(fin + (int64_t)i * n + x);
  collide_emit<R>(h, omega_of<R>(p), [&](int i, R v) { stpop<S>(fout + (int64_t)i * n + x, v); });
}

// The same step for the sites with iolet links, kStepIoletLanes lanes a
// site, lane h holding directions h, h + lanes, ... (gather, boundary value,
// collision).  Moments and collision sums run over the directions in the
// order of the per-thread code (collide_emit, and the read-back path
// iolet_fixup), so every value equals it bit for bit.  w is the lane
// group's site; a group past the end shadows site 0 and stores nothing (all
// 32 lanes take part in the shuffles).
template <typename S>
__device__ __forceinline__ void step_iolet_site(const S* __restrict__ fin, S* __restrict__ fout,
                                                const int32_t* __restrict__ src, const LinkRec* __restrict__ links,
                                                const double* __restrict__ amp, const int32_t* __restrict__ sites,
                                                int64_t nsites, const StepParams& p, int64_t w) {
  using R = typename Real<S>::type;
  constexpr int W = kStepIoletLanes, NE = (Q + W - 1) / W;
  const bool live = w < nsites;
  const int hl = threadIdx.x & (W - 1);
  const int64_t n = p.n, x = sites[live ? w : 0];
  int32_t c[NE];
  LinkRec L[NE];
  R h[NE], own[NE], a[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    c[e] = (i >= 1 && i < Q) ? src[(int64_t)(i - 1) * p.sn + x] : 0;
    // link records and amplitudes load beside the populations, not after
    // them (record 0 exists whenever a site has an iolet link)
    L[e] = links[c[e] <= -2 ? -c[e] - 2 : 0];
    h[e] = own[e] = R(0);
    if (i < Q) {
      h[e] = ldpop(fin + (i == 0 ? x : (c[e] >= 0 ? (int64_t)i * n + c[e] : (int64_t)lane_opp(i) * n + x)));
      own[e] = ldpop(fin + (int64_t)i * n + x);
    }
    a[e] = BC<R>::amp(p, amp, L[e].kind == 0 && L[e].group >= 0 ? L[e].group : 0);
  }
  // moments of the stored s'(t-1) at x, in direction order
  R d = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const R vk = __shfl_sync(FULL_MASK, own[k / W], k % W, W);
    d += vk;
    if (cx(k)) jx += cx(k) > 0 ? vk : -vk;
    if (cy(k)) jy += cy(k) > 0 ? vk : -vk;
    if (cz(k)) jz += cz(k) > 0 ? vk : -vk;
  }
  const R rho_s = R(1) + d;
  const R ux = jx / rho_s, uy = jy / rho_s, uz = jz / rho_s;
#pragma unroll
  for (int e = 0; e < NE; ++e)
    if (c[e] <= -2) h[e] = lane_iolet_value<R>(e * W + hl, L[e], h[e], rho_s, ux, uy, uz, a[e], BC<R>::val(p, L[e].iolet), p);
  // collision: sums over opposite pairs as collide_emit forms them
  const R omega = omega_of<R>(p);
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
  if (!live) return;
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    if (i < Q) stpop<S>(fout + (int64_t)i * n + x, iolet_lane_out<R>(i, h[e], bgk));
  }
}

// Pull A-B step from s'(t-1) in one launch: gather f(t) through the index
// table (walls: the site's own opposite slot), collide, store coalesced.
// Every stride-th block (the first n_iolet_blocks of them) takes iolet
// sites, 8 lanes each (step_iolet_site); the others take 256 bulk sites,
// a thread each, and leave iolet sites alone.  The iolet blocks, spread
// through the grid, run beside the bulk blocks instead of after them.
// This one-site form serves FP64 storage and the int32 table; k_step2 the
// rest.  WIDE: offsets within direction pairs (lattices above ~226M sites).
// CT: bulk codes from the compact index table (iolet lanes read the 32-bit
// one), and an L2 prefetch of the bulk tile `pf` tiles ahead.
template <typename S, bool WIDE, bool CT>
__global__ void __launch_bounds__(BLOCK, 5) k_step(const S* __restrict__ fin, S* __restrict__ fout,
                                                const IndexTables ix, const LinkRec* __restrict__ links,
                                                const double* __restrict__ amp, const int32_t* __restrict__ sites,
                                                int64_t nsites, const IoletSpread spread, uint32_t pf, uint32_t tile0,
                                                const StepParams p) {
  using R = typename Real<S>::type;
  uint32_t j;
  if (spread_block(spread, blockIdx.x, &j)) {
    pdl_wait();
    pdl_trigger();
    step_iolet_site<S>(fin, fout, ix.src, links, amp, sites, nsites, p, ((int64_t)j * BLOCK + threadIdx.x) / kStepIoletLanes);
    return;
  }
  const uint32_t n = (uint32_t)p.n, sn = (uint32_t)p.sn;
  if (tile0 == kNoTile) return;
  const uint32_t tile = tile0 + j;
  const uint32_t x = tile * BLOCK + threadIdx.x;
  if (CT && pf && threadIdx.x < 32) prefetch_tile<S, sizeof(S) >= 4, false, true>(fin, ix, n, sn, tile, pf);
  uint32_t off[Q];
  const bool live = x < n;
  // sites with an iolet link are stepped by the iolet warps
  bool skip = true;
  if (live) skip = load_offsets<CT, WIDE, LD_STREAM>(ix, sn, n, x, tile, off);
  pdl_wait();
  pdl_trigger();
  if (skip) return;
  R h[Q];
  h[0] = ldpop(fin + x);
  // fluid source: row i at s; otherwise row opp(i) at x (bounce-back)
#pragma unroll
  for (int i = 1; i < Q; ++i) h[i] = ldpop(at<WIDE>(fin, i, n, off[i]));
  collide<R>(h, omega_of<R>(p));
  if (WIDE) {
    stpop<S>(fout + x, h[0]);
#pragma unroll
    for (int i = 1; i < Q; ++i) stpop<S>(at<WIDE>(fout, i, n, slot<WIDE>(i, n, x)), h[i]);
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) stpop<S>(fout + (uint32_t)i * n + x, h[i]);
  }
}

// ---------------------------------------------------------------------------
// AA pattern.
// ---------------------------------------------------------------------------
// The sites with iolet links of an AA step at time t, W lanes a site, lane h
// holding directions h, h + W, ...: f(t) from the slots (EVEN: the site's own,
// ODD: through its codes), collision, and each post-collision population into
// the slot that its opposite direction was read from.  An iolet link's slot
// (slot i of x in both parities) gets the boundary value that the next step
// reads instead, from the moments of the stored (rounded) post-collision
// populations as the A-B gather takes them, and the mass that the link lets
// in is recorded.  No other site touches these slots, so the sites can be blocks
// of the step's own grid, every stride-th one, instead of a pass of their own
// after each step (k_aa_fix): aa_in_grid says when.  Codes, records and
// amplitudes load before the wait for the previous step; icode holds a site's
// 18 codes contiguously.
template <typename S, bool ODD>
__device__ __forceinline__ void aa_iolet_site(S* A, const int32_t* __restrict__ icode, const LinkRec* __restrict__ links,
                                              const double* __restrict__ amp, const int32_t* __restrict__ sites,
                                              int64_t nsites, const StepParams& p, double* __restrict__ lflux, int64_t q0) {
  using R = typename Real<S>::type;
  constexpr int W = kStepIoletLanes, NE = (Q + W - 1) / W;
  const bool live = q0 < nsites;
  const int64_t q = live ? q0 : 0, n = p.n;  // lanes past the end shadow site 0 and store nothing
  const int hl = threadIdx.x & (W - 1);
  const int64_t x = __ldg(sites + q);
  int32_t c[NE];
  LinkRec L[NE];
  R a[NE], h[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    c[e] = (i >= 1 && i < Q) ? __ldg(icode + q * (Q - 1) + (i - 1)) : 0;
    L[e] = links[c[e] <= -2 ? -c[e] - 2 : 0];  // record 0 exists whenever there are iolet sites
    a[e] = BC<R>::amp(p, amp, L[e].kind == 0 && L[e].group >= 0 ? L[e].group : 0);
  }
  pdl_wait();
  pdl_trigger();
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    h[e] = i < Q ? to_real(A[i == 0 ? x : (ODD ? aa_addr(i, c[e], n, x) : (int64_t)i * n + x)]) : R(0);
  }
  auto in = [&](int k) { return __shfl_sync(FULL_MASK, h[k / W], k % W, W); };
  R o[NE];  // s'_i(x), as stored
  {
    R drho = in(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int ip = 2 * k + 1;
      const R va = in(ip), vb = in(ip + 1), dp = va - vb;
      drho += va + vb;
      if (cx(ip)) jx = cx(ip) > 0 ? jx + dp : jx - dp;
      if (cy(ip)) jy = cy(ip) > 0 ? jy + dp : jy - dp;
      if (cz(ip)) jz = cz(ip) > 0 ? jz + dp : jz - dp;
    }
    const Bgk<R> b(drho, jx, jy, jz, omega_of<R>(p));
#pragma unroll
    for (int e = 0; e < NE; ++e) o[e] = e * W + hl < Q ? to_real(from_real<S>(iolet_lane_out<R>(e * W + hl, h[e], b))) : R(0);
  }
  // rho = 1 + sum s'_k, j = sum s'_k c_k in direction order
  R d = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const R vk = __shfl_sync(FULL_MASK, o[k / W], k % W, W);
    d += vk;
    if (cx(k)) jx += cx(k) > 0 ? vk : -vk;
    if (cy(k)) jy += cy(k) > 0 ? vk : -vk;
    if (cz(k)) jz += cz(k) > 0 ? vk : -vk;
  }
  const R rho = R(1) + d;
  const R ux = jx / rho, uy = jy / rho, uz = jz / rho;
  // s'_opp(i): direction i + 1 for odd i (odd lanes, W even), i - 1 for even i
  R up[NE + 1], dn[NE + 1];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    up[e] = __shfl_sync(FULL_MASK, o[e], (hl + 1) & (W - 1), W);
    dn[e + 1] = __shfl_sync(FULL_MASK, o[e], (hl + W - 1) & (W - 1), W);
  }
  up[NE] = dn[0] = R(0);
  if (!live) return;
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    if (i >= Q) continue;
    if (i == 0) {
      stpop<S>(A + x, o[0]);
      continue;
    }
    R v = (i & 1) ? (hl == W - 1 ? up[e + 1] : up[e]) : (hl == 0 ? dn[e] : dn[e + 1]);
    if (c[e] <= -2) {
      const R val = lane_iolet_value<R>(i, L[e], v, rho, ux, uy, uz, a[e], BC<R>::val(p, L[e].iolet), p);
      lflux[-c[e] - 2] = (double)val - (double)v;
      v = val;
    }
    stpop<S>(A + (ODD ? aa_addr(i, c[e], n, x) : (int64_t)i * n + x), v);
  }
}

// The iolet blocks of an AA step's grid (GRID; otherwise the bulk blocks take
// all sites and k_aa_fix follows).
struct AAIolets {
  const int32_t* icode;
  const LinkRec* links;
  const double* amp;
  const int32_t* sites;
  int64_t nsites;
  const uint32_t* imask;
  double* lflux;
  unsigned blocks;  // iolet blocks, every stride-th of the grid's first ones
  BlockDiv stride;
};
// True for an iolet block, whose sites it steps; otherwise *bulk is the bulk block's number.
template <typename S, bool ODD, bool GRID>
__device__ __forceinline__ bool aa_iolet_block(S* A, const AAIolets& io, const StepParams& p, uint32_t* bulk) {
  if (!GRID) {
    *bulk = blockIdx.x;
    return false;
  }
  const unsigned b = blockIdx.x, j = block_div(b, io.stride);
  *bulk = b - min(io.blocks, j + 1);
  if (b != j * io.stride.d || j >= io.blocks) return false;
  aa_iolet_site<S, ODD>(A, io.icode, io.links, io.amp, io.sites, io.nsites, p, io.lflux,
                               ((int64_t)j * blockDim.x + threadIdx.x) / kStepIoletLanes);
  return true;
}
// Whether the iolet blocks step site x.
template <bool GRID>
__device__ __forceinline__ bool left_to_iolets(const AAIolets& io, uint32_t x) {
  return GRID && ((__ldg(io.imask + (x >> 5)) >> (x & 31)) & 1u);
}

// Even step: f(t) in place -> collide -> s'(t) stored swapped (slot ibar).
template <typename S, bool GRID>
__global__ void __launch_bounds__(BLOCK) k_aa_even(S* A, const AAIolets io, const StepParams p) {
  using R = typename Real<S>::type;
  uint32_t bulk;
  if (aa_iolet_block<S, false, GRID>(A, io, p, &bulk)) return;
  const int64_t n = p.n;
  const int64_t x = (int64_t)bulk * BLOCK + threadIdx.x;
  const bool skip = x >= n || left_to_iolets<GRID>(io, (uint32_t)x);
  pdl_wait();
  pdl_trigger();
  if (skip) return;
  R h[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) h[i] = to_real(A[(int64_t)i * n + x]);
  collide<R>(h, omega_of<R>(p));
#pragma unroll
  for (int i = 0; i < Q; ++i) stpop<S>(A + (int64_t)opp(i) * n + x, h[i]);
}

// Even step for 16-bit storage, two neighbouring sites per thread with 4-byte
// accesses (rows are 4-byte aligned when n is even).  The two collisions run
// in paired FP32 instructions (collide2), which halves the arithmetic
// instructions of a kernel whose 16-bit traffic leaves instruction issue as
// a limit.  Four blocks per SM (64 registers, a few bytes of spill) measured
// 4-5 % faster than the scalar collisions, and than three blocks without
// the spill.
template <typename S> struct Pair;
template <> struct Pair<__nv_bfloat16> {
  using T = __nv_bfloat162;
  static __device__ __forceinline__ float2 to(T v) { return __bfloat1622float2(v); }
  static __device__ __forceinline__ T from(float a, float b) { return __floats2bfloat162_rn(a, b); }
};
template <> struct Pair<__half> {
  using T = __half2;
  static __device__ __forceinline__ float2 to(T v) { return __half22float2(v); }
  static __device__ __forceinline__ T from(float a, float b) { return __floats2half2_rn(a, b); }
};
template <> struct Pair<float> {
  using T = float2;
  static __device__ __forceinline__ float2 to(T v) { return v; }
  static __device__ __forceinline__ T from(float a, float b) { return make_float2(a, b); }
};

// Paired FP32 arithmetic (sm_100 and later): one instruction applies the
// operation to .x and .y, each rounded as the scalar operation is.
__device__ __forceinline__ float2 p_splat(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// collide() of two sites at once, h[i] = (site x, site x + 1).  Directions
// 2p-1 and 2p are opposite, so each pair shares c.u and 4.5 (c.u)^2 - 1.5 u.u
// and differs only in the sign of the 3 c.u term.
__device__ __forceinline__ void collide2(float2* h, float omega) {
  float2 d = h[0];
#pragma unroll
  for (int i = 1; i < Q; ++i) d = p_add(d, h[i]);
  // momentum: each component is the sum over the pairs that move along it
  float2 jx = p_sub(h[1], h[2]), jy = p_sub(h[3], h[4]), jz = p_sub(h[5], h[6]);
#pragma unroll
  for (int i = 7; i < Q; ++i) {
    if (cx(i)) jx = cx(i) > 0 ? p_add(jx, h[i]) : p_sub(jx, h[i]);
    if (cy(i)) jy = cy(i) > 0 ? p_add(jy, h[i]) : p_sub(jy, h[i]);
    if (cz(i)) jz = cz(i) > 0 ? p_add(jz, h[i]) : p_sub(jz, h[i]);
  }
  const float2 rho = p_add(p_splat(1.f), d);
  const float2 inv = make_float2(1.f / rho.x, 1.f / rho.y);
  const float2 ux = p_mul(jx, inv), uy = p_mul(jy, inv), uz = p_mul(jz, inv);
  const float2 nusq = p_mul(p_splat(-1.5f), p_fma(uz, uz, p_fma(uy, uy, p_mul(ux, ux))));
  const float2 om = p_splat(omega);
  {  // rest population: c.u = 0
    const float2 heq = p_mul(p_splat(1.f / 3.f), p_fma(rho, nusq, d));
    h[0] = p_fma(om, p_sub(heq, h[0]), h[0]);
  }
#pragma unroll
  for (int q = 1; q < 10; ++q) {
    const int i = 2 * q - 1;  // c_i has a positive first nonzero component
    float2 cu = cx(i) ? ux : uy;
    if (cx(i) && cy(i)) cu = cy(i) > 0 ? p_add(ux, uy) : p_sub(ux, uy);
    if (cx(i) && cz(i)) cu = cz(i) > 0 ? p_add(ux, uz) : p_sub(ux, uz);
    if (!cx(i) && cz(i)) cu = cy(i) ? (cz(i) > 0 ? p_add(uy, uz) : p_sub(uy, uz)) : uz;
    const float2 a = p_fma(p_mul(p_splat(4.5f), cu), cu, nusq);
    const float2 tp = p_fma(p_splat(3.f), cu, a), tm = p_fma(p_splat(-3.f), cu, a);
    const float2 w = p_splat(wgt<float>(i));
    const float2 ep = p_mul(w, p_fma(rho, tp, d)), em = p_mul(w, p_fma(rho, tm, d));
    h[i] = p_fma(om, p_sub(ep, h[i]), h[i]);
    h[i + 1] = p_fma(om, p_sub(em, h[i + 1]), h[i + 1]);
  }
}

template <typename S>
__global__ void __launch_bounds__(BLOCK, 4) k_aa_even2(S* A, const StepParams p) {
  using P = Pair<S>;
  using T = typename P::T;
  const int64_t n = p.n;
  const int64_t x = 2 * ((int64_t)blockIdx.x * BLOCK + threadIdx.x);
  pdl_wait();
  pdl_trigger();
  if (x >= n) return;
  T* A2 = reinterpret_cast<T*>(A);
  const int64_t n2 = n / 2, x2 = x / 2;
  float2 h[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) h[i] = P::to(A2[(int64_t)i * n2 + x2]);
  collide2(h, p.omegaf);
#pragma unroll
  for (int i = 0; i < Q; ++i) __stcs(A2 + (int64_t)opp(i) * n2 + x2, P::from(h[i].x, h[i].y));
}

// collide_emit() of two sites at once, h[i] = (site x, site x + 1): the same
// operations in the same order, each pair of scalar operations one paired
// FP32 instruction (rounded as the scalar one), so each site gets the bits
// of the per-thread collision.
__device__ __forceinline__ float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 p_cdotu(int i, float2 ux, float2 uy, float2 uz) {
  float2 s = p_splat(0.f);
  if (cx(i)) s = p_add(s, cx(i) > 0 ? ux : p_neg(ux));
  if (cy(i)) s = p_add(s, cy(i) > 0 ? uy : p_neg(uy));
  if (cz(i)) s = p_add(s, cz(i) > 0 ? uz : p_neg(uz));
  return s;
}
template <typename Emit>
__device__ __forceinline__ void collide_pair(const float2* h, float omega, Emit&& emit) {
  float2 drho = h[0], jx = p_splat(0.f), jy = p_splat(0.f), jz = p_splat(0.f);
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const int i = 2 * p + 1;
    const float2 sp = p_add(h[i], h[i + 1]), dp = p_sub(h[i], h[i + 1]);
    drho = p_add(drho, sp);
    if (cx(i)) jx = cx(i) > 0 ? p_add(jx, dp) : p_sub(jx, dp);
    if (cy(i)) jy = cy(i) > 0 ? p_add(jy, dp) : p_sub(jy, dp);
    if (cz(i)) jz = cz(i) > 0 ? p_add(jz, dp) : p_sub(jz, dp);
  }
  const float2 rho = p_add(p_splat(1.f), drho);
  const float2 inv = make_float2(1.f / rho.x, 1.f / rho.y);
  const float2 ux = p_mul(jx, inv), uy = p_mul(jy, inv), uz = p_mul(jz, inv);
  const float2 usq15 = p_mul(p_splat(1.5f), p_fma(uz, uz, p_fma(uy, uy, p_mul(ux, ux))));
  const float2 om1 = p_splat(1.f - omega);
  float2 wr[3], wd[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float ow = omega * wgt<float>(c == 0 ? 0 : (c == 1 ? 1 : 7));
    wr[c] = p_mul(p_splat(ow), rho);
    wd[c] = p_mul(p_splat(ow), drho);
  }
  emit(0, p_fma(om1, h[0], p_fma(p_neg(wr[0]), usq15, wd[0])));
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const int i = 2 * p + 1, c = i <= 6 ? 1 : 2;
    const float2 cu = p_cdotu(i, ux, uy, uz);
    const float2 a = p_fma(p_mul(p_splat(4.5f), cu), cu, p_neg(usq15));
    emit(i, p_fma(om1, h[i], p_fma(wr[c], p_fma(p_splat(3.f), cu, a), wd[c])));
    emit(i + 1, p_fma(om1, h[i + 1], p_fma(wr[c], p_fma(p_splat(-3.f), cu, a), wd[c])));
  }
}

// Two sites a thread on the compact table (k_step2, k_aa_odd2): thread t of a
// block takes sites x = 64 (t / 32) + t % 32 and x + 32 of the block's tile, so
// every load and store of a warp stays one run of 32 sites.
__device__ __forceinline__ uint32_t pair_site(uint32_t tile) {
  return tile * CT_TILE + 2 * (threadIdx.x & ~31u) + (threadIdx.x & 31u);
}
// Row-form words of the pair's sites (y = x + 32 may lie past the end: x's then).
__device__ __forceinline__ void load_pair_words(const IndexTables& ix, bool wide, uint32_t sn, uint32_t x, uint32_t y,
                                                uint32_t* wa, uint32_t* wb) {
#pragma unroll
  for (int q = 0; q < CT_ROW_WORDS; ++q) {
    const uint32_t* row = wide ? ix.rtab + (uint64_t)q * sn : ix.rtab + (uint32_t)q * sn;
    wa[q] = __ldg(row + x);
    wb[q] = __ldg(row + y);
  }
}
// Offset that direction i of site x is read from (pull), or read from and
// written to (AAODD), given its row-form mask and positions.
template <bool WIDE, bool AAODD>
__device__ __forceinline__ uint32_t row_offset(int i, uint32_t mask, const uint32_t* pos, uint32_t n) {
  const uint32_t s = pos[row_group(i)] - (uint32_t)cx(i);
  return ((mask >> (i - 1)) & 1u) ? slot<WIDE>(AAODD ? opp(i) : i, n, s) : slot<WIDE>(AAODD ? i : opp(i), n, pos[CT_GROUPS]);
}

// Offset-form words of the pair's sites, and the offset that direction i of
// site x is read from (pull), given the tile's base of the direction.
__device__ __forceinline__ void load_pair_offsets(const IndexTables& ix, bool wide, uint32_t sn, uint32_t x, uint32_t y,
                                                  uint32_t* wa, uint32_t* wb) {
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const uint32_t* row = wide ? ix.ctab + (uint64_t)q * sn : ix.ctab + (uint32_t)q * sn;
    wa[q] = __ldg(row + x);
    wb[q] = __ldg(row + y);
  }
}
template <bool WIDE>
__device__ __forceinline__ uint32_t pair_offset(int i, const uint32_t* w, uint32_t base, uint32_t n, uint32_t x) {
  const uint32_t o = offset_of(w, i);
  return o < CT_IOLET ? slot<WIDE>(i, n, base + o) : slot<WIDE>(opp(i), n, x);
}
__device__ __forceinline__ bool has_iolet(const IndexTables& ix, uint32_t x) {
  return (__ldg(ix.imask + (x >> 5)) >> (x & 31)) & 1u;
}

// Pull A-B step (k_step) with two sites a thread, FP32 or 16-bit storage on the
// compact table, any number of sites.  Bound by DRAM in FP32 (164 bytes a
// site with the row-form index) and by instruction issue and latency in 16
// bits.  Pairing halves the arithmetic: the two collisions run in paired FP32
// instructions (collide_pair: the bits of k_step).  The pair is x and x + 32,
// not two neighbours: a warp's gather of neighbours spans 64 sites in steps
// of two, twice the sectors a request, and needs an even site count for its
// vector stores.  20M-site tree, per step: FP32 563 -> 495 us, BF16 406 -> 345
// us against neighbours on the 16-bit offset table; 2.0M sites (odd) FP32 66.5
// -> 56.4 us, BF16 47.7 -> 38.7 us against one site a thread on it.
// Prefetch 3 tiles per SM ahead: FP32 495 us with the gathered rows, 500
// without them, 516 with no prefetch, 537 at 6; 16-bit storage prefetches
// the index words only.  A tile in offset form takes its two sites at once as
// well (TILE_PAIRS; pair_tiles says when), or one after the other.
template <typename S, bool WIDE, bool TILE_PAIRS>
__global__ void __launch_bounds__(PAIR, pair_blocks<S>()) k_step2(const S* __restrict__ fin, S* __restrict__ fout,
                                                const IndexTables ix, const LinkRec* __restrict__ links,
                                                const double* __restrict__ amp, const int32_t* __restrict__ sites,
                                                int64_t nsites, const IoletSpread spread, uint32_t pf, uint32_t tile0,
                                                const StepParams p) {
  uint32_t j;
  if (spread_block(spread, blockIdx.x, &j)) {
    pdl_wait();
    pdl_trigger();
    step_iolet_site<S>(fin, fout, ix.src, links, amp, sites, nsites, p, ((int64_t)j * PAIR + threadIdx.x) / kStepIoletLanes);
    return;
  }
  const uint32_t n = (uint32_t)p.n, sn = (uint32_t)p.sn;
  if (tile0 == kNoTile) return;
  const uint32_t tile = tile0 + j;
  const uint32_t x = pair_site(tile), y = x + 32;
  if (pf && threadIdx.x < 32) prefetch_tile<S, sizeof(S) == 4, false, TILE_PAIRS>(fin, ix, n, sn, tile, pf);
  int32_t bs[CT_GROUPS];
  if (load_row_bases(ix, tile, bs)) {
    const uint32_t y1 = y < n ? y : x;  // a thread without a second site repeats its first, and does not store it
    uint32_t wa[CT_ROW_WORDS], wb[CT_ROW_WORDS];
    if (x < n) load_pair_words(ix, WIDE, sn, x, y1, wa, wb);
    pdl_wait();
    pdl_trigger();
    if (x >= n) return;
    const bool da = !((wa[0] >> CT_IOLET_BIT) & 1u), db = y < n && !((wb[0] >> CT_IOLET_BIT) & 1u);
    uint32_t pa[CT_GROUPS + 1], pb[CT_GROUPS + 1];
    row_positions(x, bs, wa[1], wa[2], pa);
    row_positions(y1, bs, wb[1], wb[2], pb);
    float2 h[Q];
    h[0] = make_float2(ldpop(fin + x), ldpop(fin + y1));
#pragma unroll
    for (int i = 1; i < Q; ++i)
      h[i] = make_float2(ldpop(at<WIDE>(fin, i, n, row_offset<WIDE, false>(i, wa[0], pa, n))),
                         ldpop(at<WIDE>(fin, i, n, row_offset<WIDE, false>(i, wb[0], pb, n))));
    collide_pair(h, p.omegaf, [&](int i, float2 v) {
      S* o = i == 0 ? fout + x : at<WIDE>(fout, i, n, slot<WIDE>(i, n, x));
      if (da) stpop<S>(o, v.x);
      if (db) stpop<S>(o + 32, v.y);
    });
    return;
  }
  if (TILE_PAIRS) {
    const uint32_t y1 = y < n ? y : x;
    uint32_t wa[9], wb[9];
    bool da = false, db = false;
    if (x < n) {
      load_pair_offsets(ix, WIDE, sn, x, y1, wa, wb);
      da = !has_iolet(ix, x);
      db = y < n && !has_iolet(ix, y);
    }
    pdl_wait();
    pdl_trigger();
    if (x >= n) return;
    const int32_t* tb = ix.tbase + (uint64_t)tile * CT_BASES;
    float2 h[Q];
    h[0] = make_float2(ldpop(fin + x), ldpop(fin + y1));
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const uint32_t base = (uint32_t)__ldg(tb + i - 1);
      h[i] = make_float2(ldpop(at<WIDE>(fin, i, n, pair_offset<WIDE>(i, wa, base, n, x))),
                         ldpop(at<WIDE>(fin, i, n, pair_offset<WIDE>(i, wb, base, n, y1))));
    }
    collide_pair(h, p.omegaf, [&](int i, float2 v) {
      S* o = i == 0 ? fout + x : at<WIDE>(fout, i, n, slot<WIDE>(i, n, x));
      if (da) stpop<S>(o, v.x);
      if (db) stpop<S>(o + 32, v.y);
    });
    return;
  }
  for (uint32_t z = x; z < n && z <= y; z += 32) {
    uint32_t off[Q];
    offset_links<WIDE, LD_NC>(ix, sn, z, tile, [&](int i, bool fluid, uint32_t s) {
      off[i] = fluid ? slot<WIDE>(i, n, s) : slot<WIDE>(opp(i), n, z);
    });
    pdl_wait();
    if (has_iolet(ix, z)) continue;
    float h[Q];
    h[0] = ldpop(fin + z);
#pragma unroll
    for (int i = 1; i < Q; ++i) h[i] = ldpop(at<WIDE>(fin, i, n, off[i]));
    collide<float>(h, p.omegaf);
    stpop<S>(fout + z, h[0]);
#pragma unroll
    for (int i = 1; i < Q; ++i) stpop<S>(at<WIDE>(fout, i, n, slot<WIDE>(i, n, z)), h[i]);
  }
  pdl_trigger();
}

// Boundary value of iolet link (pull direction i, record L) at a site whose
// pre-collision moments at time t are (drho, u) and whose outgoing
// post-collision population is `out` (= s'_ibar): incoming f_i(t+1) - w_i.
template <typename R>
__device__ __forceinline__ R iolet_value(int i, const LinkRec& L, R out, R rho, R ux, R uy, R uz,
                                         const double* __restrict__ amp, const StepParams& p) {
  const IoletParam& io = p.io[L.iolet];
  if (L.kind == 0) {
    R r = p.ladd_rho_one ? R(1) : rho;
    return out + BC<R>::coef(L) * r * BC<R>::amp(p, amp, L.group) * BC<R>::val(p, L.iolet);
  }
  R gx = ux, gy = uy, gz = uz;
  if (!p.ghost_full_u) {
    R un = dot3(gx, gy, gz, BC<R>::nx(io), BC<R>::ny(io), BC<R>::nz(io));
    gx = un * BC<R>::nx(io);
    gy = un * BC<R>::ny(io);
    gz = un * BC<R>::nz(io);
  }
  R drho = BC<R>::val(p, L.iolet);
  return ghost_heq<R>(wgt<R>(i), drho, cdotu<R>(i, gx, gy, gz), dot3(gx, gy, gz, gx, gy, gz));
}

// After an AA step at time t: overwrite the slots that the iolet links of
// each iolet site read in the next step with their boundary values, and
// record the mass each link lets in.  A lane's codes, stored values and (iolet
// links) link records are one load each, so the pass is a few rounds of
// loads whatever the site's number of iolet links; records and amplitudes
// load before the wait for the step kernel.  The site's stored post-collision
// populations s'_ibar(x) sit in slot i of x after an even step, and in the
// slot it read direction i from after an odd step; an iolet link's slot is
// slot i of x in both cases.  Boundary values use the moments of these
// stored values, as the A-B gather does, summed over s'_0, s'_1, ... in the
// order of the A-B warp path, so the two schemes give the same bits.
// icode[q][i - 1] is the index code of direction i at iolet site q: 72
// contiguous bytes a site.  Two iolet sites a warp: 16 lanes a site, lane h
// holding direction h and, for h < 3, also direction 16 + h (32 registers,
// 8 blocks per SM).  Against one warp a site it runs in half the warps: the
// 54k iolet sites of the 20M-site tree in 2.8 waves instead of 5.6, about
// 3 us less a step.
template <typename S, bool ODD>
__global__ void __launch_bounds__(256, 8) k_aa_fix(S* A, const int32_t* __restrict__ icode,
                                                 const LinkRec* __restrict__ links, const double* __restrict__ amp,
                                                 const int32_t* __restrict__ sites, int64_t nsites,
                                                 const StepParams p, double* __restrict__ lflux) {
  using R = typename Real<S>::type;
  constexpr int W = kFixLanes, NE = (Q + W - 1) / W;
  const int64_t q0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / W;
  const bool live = q0 < nsites;
  const int64_t q = live ? q0 : 0;  // lanes past the end shadow site 0 and store nothing
  const int hl = threadIdx.x & (W - 1);
  const int64_t x = __ldg(sites + q);
  int32_t c[NE];
  LinkRec L[NE];
  R a[NE], v[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    c[e] = (i >= 1 && i < Q) ? __ldg(icode + q * (Q - 1) + (i - 1)) : 0;
    // link records and amplitudes do not change between steps: loaded before
    // the wait for the step kernel (record 0 exists whenever there are iolet sites)
    L[e] = links[c[e] <= -2 ? -c[e] - 2 : 0];
    a[e] = BC<R>::amp(p, amp, L[e].kind == 0 && L[e].group >= 0 ? L[e].group : 0);
  }
  pdl_wait();
  pdl_trigger();
  const int64_t n = p.n;
  // s'_ibar(x): the value in the slot the link of direction i reads
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    v[e] = R(0);
    if (i < Q) v[e] = to_real(A[i == 0 ? x : (ODD ? aa_addr(i, c[e], n, x) : (int64_t)i * n + x)]);
  }
  // rho = 1 + sum s'_k, j = sum s'_k c_k in direction order; s'_k sits with direction opp(k)
  R d = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const int o = opp(k);
    const R vk = __shfl_sync(FULL_MASK, v[o / W], o % W, W);
    d += vk;
    if (cx(k)) jx += cx(k) > 0 ? vk : -vk;
    if (cy(k)) jy += cy(k) > 0 ? vk : -vk;
    if (cz(k)) jz += cz(k) > 0 ? vk : -vk;
  }
  const R rho = R(1) + d;
  const R ux = jx / rho, uy = jy / rho, uz = jz / rho;
  if (!live) return;
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = e * W + hl;
    if (c[e] <= -2) {
      const R val = lane_iolet_value<R>(i, L[e], v[e], rho, ux, uy, uz, a[e], BC<R>::val(p, L[e].iolet), p);
      lflux[-c[e] - 2] = (double)val - (double)v[e];
      A[(int64_t)i * n + x] = from_real<S>(val);
    }
  }
}

// Odd step: gather f(t) through the index table, collide, and write each
// post-collision population into the slot it came from, where the site
// downstream (or, across a wall or iolet, the site itself) reads it in the
// next (even) step.  Sites with iolet links: aa_iolet_site or k_aa_fix.
// This one-site form serves FP64 storage, the int32 table, small 16-bit
// lattices (kOddPairSites) and, in 16 bits or from kOffsetPairSites on, those
// whose tiles mostly have the offset form (2.0M sites in (x, y, z) order, BF16:
// 41 us; k_aa_odd2 44, and 47 with both sites at once, which spills); k_aa_odd2
// the rest.  The 18 slot offsets (32-bit) are computed once and held in registers
// for the stores, so the index row is read once.  WIDE: offsets within
// direction pairs (lattices above ~226M sites), four blocks per SM instead
// of five.  CT: codes from the compact index table, and the first warp
// prefetches into L2 the tile `pf` blocks ahead (0: none).
template <typename S, bool WIDE, bool CT>
__global__ void __launch_bounds__(BLOCK, WIDE ? 4 : 5) k_aa_odd(S* A, const IndexTables ix, uint32_t pf,
                                                               const StepParams p) {
  using R = typename Real<S>::type;
  const uint32_t n = (uint32_t)p.n, sn = (uint32_t)p.sn;
  const uint32_t x = blockIdx.x * BLOCK + threadIdx.x;
  if (CT && pf && threadIdx.x < 32) prefetch_tile<S, sizeof(S) >= 4, true, true>(A, ix, n, sn, blockIdx.x, pf);
  int32_t code[Q];
  if (x < n) load_codes<CT, WIDE, LD_NC>(ix, sn, x, blockIdx.x, code);
  pdl_wait();
  pdl_trigger();
  if (x >= n) return;
  uint32_t off[Q];
  R h[Q];
  h[0] = to_real(A[x]);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    // slot opp(i) of the source, or slot i of x itself across a wall or iolet
    off[i] = code[i] >= 0 ? slot<WIDE>(opp(i), n, (uint32_t)code[i]) : slot<WIDE>(i, n, x);
    h[i] = to_real(*at<WIDE>(A, i, n, off[i]));
  }
  collide<R>(h, omega_of<R>(p));
  stpop<S>(A + x, h[0]);
#pragma unroll
  for (int i = 1; i < Q; ++i) stpop<S>(at<WIDE>(A, i, n, off[i]), h[opp(i)]);
}

// The odd step with two sites a thread (k_step2's pairing: x and x + 32), FP32 or
// 16-bit storage on the compact table.  A site's offsets follow from three
// index words, so they are formed twice, for the gather and for the stores,
// instead of being held across the collision in 36 registers: that is what
// lets two sites share a thread at 80 (72) registers.  20M-site tree, step
// with the iolet pass: FP32 597 -> 532 us, BF16 460 -> 388 us; 2.0M sites FP32
// 75 -> 67, BF16 58 -> 48 us.
template <typename S, bool WIDE, bool GRID>
__global__ void __launch_bounds__(PAIR, pair_blocks<S>()) k_aa_odd2(S* A, const IndexTables ix, const AAIolets io, uint32_t pf,
                                                                        const StepParams p) {
  uint32_t tile;
  if (aa_iolet_block<S, true, GRID>(A, io, p, &tile)) return;
  const uint32_t n = (uint32_t)p.n, sn = (uint32_t)p.sn;
  const uint32_t x = pair_site(tile), y = x + 32;
  if (pf && threadIdx.x < 32) prefetch_tile<S, sizeof(S) == 4, true, false>(A, ix, n, sn, tile, pf);
  int32_t bs[CT_GROUPS];
  if (load_row_bases(ix, tile, bs)) {
    const uint32_t y1 = y < n ? y : x;  // a thread without a second site repeats its first, and does not store it
    uint32_t wa[CT_ROW_WORDS], wb[CT_ROW_WORDS];
    if (x < n) load_pair_words(ix, WIDE, sn, x, y1, wa, wb);
    pdl_wait();
    pdl_trigger();
    if (x >= n) return;
    constexpr uint32_t iolet = GRID ? 1u << CT_IOLET_BIT : 0u;
    const bool da = !(wa[0] & iolet), db = y < n && !(wb[0] & iolet);
    uint32_t pa[CT_GROUPS + 1], pb[CT_GROUPS + 1];
    row_positions(x, bs, wa[1], wa[2], pa);
    row_positions(y1, bs, wb[1], wb[2], pb);
    float2 h[Q];
    h[0] = make_float2(to_real(A[x]), to_real(A[y1]));
#pragma unroll
    for (int i = 1; i < Q; ++i)
      h[i] = make_float2(to_real(*at<WIDE>(A, i, n, row_offset<WIDE, true>(i, wa[0], pa, n))),
                         to_real(*at<WIDE>(A, i, n, row_offset<WIDE, true>(i, wb[0], pb, n))));
    float2 o[Q];
    collide_pair(h, p.omegaf, [&](int i, float2 v) { o[i] = v; });
    // the offsets again, from the words: held across the collision they would cost 36 registers
#pragma unroll
    for (int q = 0; q < CT_ROW_WORDS; ++q) asm volatile("" : "+r"(wa[q]), "+r"(wb[q]));
    load_row_bases(ix, tile, bs);
    row_positions(x, bs, wa[1], wa[2], pa);
    row_positions(y, bs, wb[1], wb[2], pb);
    if (da) stpop<S>(A + x, o[0].x);
    if (db) stpop<S>(A + y, o[0].y);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if (da) stpop<S>(at<WIDE>(A, i, n, row_offset<WIDE, true>(i, wa[0], pa, n)), o[opp(i)].x);
      if (db) stpop<S>(at<WIDE>(A, i, n, row_offset<WIDE, true>(i, wb[0], pb, n)), o[opp(i)].y);
    }
    return;
  }
  pdl_wait();
  pdl_trigger();
  for (uint32_t z = x; z < n && z <= y; z += 32) {
    if (left_to_iolets<GRID>(io, z)) continue;
    int32_t code[Q];
    offset_links<WIDE, LD_NC>(ix, sn, z, tile, [&](int i, bool fluid, uint32_t s) { code[i] = fluid ? (int32_t)s : -1; });
    uint32_t off[Q];
    float h[Q];
    h[0] = to_real(A[z]);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      off[i] = code[i] >= 0 ? slot<WIDE>(opp(i), n, (uint32_t)code[i]) : slot<WIDE>(i, n, z);
      h[i] = to_real(*at<WIDE>(A, i, n, off[i]));
    }
    collide<float>(h, p.omegaf);
    stpop<S>(A + z, h[0]);
#pragma unroll
    for (int i = 1; i < Q; ++i) stpop<S>(at<WIDE>(A, i, n, off[i]), h[opp(i)]);
  }
}

// ---------------------------------------------------------------------------
// Compact index table (layout in hlb_common.cuh), built once from the 32-bit
// table: one block per tile.  A thread loads its site's 18 codes, and the
// block finds whether the row form holds for all of its sites (a source of
// the own row at x - cx, one position a group, spans of 8 bits) and the
// groups' bases.  Otherwise the block writes the offset form: per direction
// the smallest and largest fluid source (warp min/max, then across the eight
// warps), the base, and each thread its offset; pairs of directions share a
// word.  Padding entries (n <= x < sn) read as walls.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(CT_TILE, 3) k_ctab_build(const int32_t* __restrict__ src, int64_t n, int64_t sn,
                                                        uint32_t* __restrict__ ctab, int32_t* __restrict__ tbase,
                                                        uint32_t* __restrict__ rtab, int32_t* __restrict__ rbase,
                                                        int32_t* __restrict__ misfit) {
  static_assert(CT_TILE == 256, "eight warps a tile");
  __shared__ uint32_t smin[8], smax[8];
  __shared__ int32_t gmin[8][CT_GROUPS], gmax[8][CT_GROUPS];
  const int64_t x = (int64_t)blockIdx.x * CT_TILE + threadIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t s[Q];
#pragma unroll
  for (int i = 1; i < Q; ++i) s[i] = x < n ? src[(int64_t)(i - 1) * sn + x] : -1;
  // row form: per group the position p = s + cx less x
  constexpr int32_t NONE = INT32_MAX;
  uint32_t mask = 0;
  int32_t d[CT_GROUPS];
#pragma unroll
  for (int g = 0; g < CT_GROUPS; ++g) d[g] = NONE;
  bool rows = true;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (s[i] <= -2) mask |= 1u << CT_IOLET_BIT;
    if (s[i] < 0) continue;
    mask |= 1u << (i - 1);
    const int32_t v = (int32_t)((int64_t)s[i] + cx(i) - x);
    const int g = row_group(i);
    if (g == CT_GROUPS) {
      rows &= v == 0;
    } else {
      rows &= d[g] == NONE || d[g] == v;
      d[g] = v;
    }
  }
#pragma unroll
  for (int g = 0; g < CT_GROUPS; ++g) {
    const int32_t lo = __reduce_min_sync(FULL_MASK, d[g]), hi = __reduce_max_sync(FULL_MASK, d[g] == NONE ? INT32_MIN : d[g]);
    if (lane == 0) {
      gmin[wid][g] = lo;
      gmax[wid][g] = hi;
    }
  }
  rows = __syncthreads_and(rows);
  int32_t base[CT_GROUPS];
#pragma unroll
  for (int g = 0; g < CT_GROUPS; ++g) {
    int32_t lo = gmin[0][g], hi = gmax[0][g];
    for (int k = 1; k < 8; ++k) {
      lo = min(lo, gmin[k][g]);
      hi = max(hi, gmax[k][g]);
    }
    base[g] = lo == NONE ? 0 : lo;  // no site of the tile has a fluid source in the group
    rows &= lo == NONE || (int64_t)hi - lo <= 255;
  }
  if (threadIdx.x < CT_GROUPS) {
    int32_t v = CT_NO_ROWS;
#pragma unroll
    for (int g = 0; g < CT_GROUPS; ++g)
      if (rows && (int)threadIdx.x == g) v = base[g];
    rbase[(int64_t)blockIdx.x * CT_GROUPS + threadIdx.x] = v;
  }
  if (rows) {  // uniform over the block
    uint32_t w[2] = {0u, 0u};
#pragma unroll
    for (int g = 0; g < CT_GROUPS; ++g)
      if (d[g] != NONE) w[g / 4] |= (uint32_t)(d[g] - base[g]) << (8 * (g % 4));
    if (x < sn) {
      rtab[x] = mask;
      rtab[sn + x] = w[0];
      rtab[2 * sn + x] = w[1];
    }
    return;
  }
  uint32_t word = 0;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    uint32_t lo = __reduce_min_sync(FULL_MASK, s[i] >= 0 ? (uint32_t)s[i] : 0xffffffffu);
    uint32_t hi = __reduce_max_sync(FULL_MASK, s[i] >= 0 ? (uint32_t)s[i] : 0u);
    if (lane == 0) {
      smin[wid] = lo;
      smax[wid] = hi;
    }
    __syncthreads();
    lo = smin[0];
    hi = smax[0];
    for (int k = 1; k < 8; ++k) {
      lo = min(lo, smin[k]);
      hi = max(hi, smax[k]);
    }
    __syncthreads();
    const bool any = lo != 0xffffffffu;  // some site of the tile has a fluid source
    const uint32_t b = any ? lo : 0u;
    if (threadIdx.x == 0) {
      tbase[(int64_t)blockIdx.x * CT_BASES + (i - 1)] = (int32_t)b;
      if (any && hi - lo > CT_MAX_SPAN) atomicOr(misfit, 1);
      if (i == 1) atomicAdd(misfit + 1, 1);
    }
    const uint32_t o = s[i] >= 0 ? ((uint32_t)s[i] - b) & 0xffffu : (s[i] == -1 ? CT_WALL : CT_IOLET);
    if (i & 1) {
      word = o;
    } else {
      word |= o << 16;
      if (x < sn) ctab[(int64_t)(i / 2 - 1) * sn + x] = word;
    }
  }
  if (threadIdx.x < CT_BASES - (Q - 1)) tbase[(int64_t)blockIdx.x * CT_BASES + (Q - 1) + threadIdx.x] = 0;
}

// ---------------------------------------------------------------------------
// Read-back kernels.
// ---------------------------------------------------------------------------
// Density, velocity and wall shear stress of f(t).  Bound by DRAM: 76 bytes of
// FP32 populations and 20 of output a site, and of the index the row form's
// mask word tells wall links (4 bytes; the gathers 12) where the int32 table
// took 72, twice in the gather modes.  20.0M sites, FP32, f(t) in place: 563 ->
// 406 us; FP64, 200k sites: 189 -> 128 us (see the zero terms below).
template <typename S, int MODE, bool CT>
__global__ void __launch_bounds__(READ) k_macros(const S* __restrict__ fin, const IndexTables ix,
                                                 const LinkRec* __restrict__ links, const double* __restrict__ amp,
                                                 const float* __restrict__ normal, const StepParams p,
                                                 float* __restrict__ rho_out, float* __restrict__ u_out,
                                                 float* __restrict__ wss_out) {
  using R = typename Real<S>::type;
  const int64_t n = p.n;
  const int64_t x = (int64_t)blockIdx.x * READ + threadIdx.x;
  if (x >= n) return;
  const uint32_t tile = (uint32_t)(x / CT_TILE);
  R h[Q];
  uint32_t wall = 0;  // directions with a wall link
  if (wss_out) {
    wall = ~load_state<S, MODE, CT, true>(fin, ix, links, amp, p, x, tile, h) & ((1u << (Q - 1)) - 1u);
    if (wall && ((__ldg(ix.imask + (x >> 5)) >> (x & 31)) & 1u)) {  // some of them iolet links
#pragma unroll
      for (int i = 1; i < Q; ++i)
        if (((wall >> (i - 1)) & 1u) && ix.src[(int64_t)(i - 1) * p.sn + x] != -1) wall &= ~(1u << (i - 1));
    }
  } else {
    load_state<S, MODE, CT, false>(fin, ix, links, amp, p, x, tile, h);
  }
  Macro<R> m = moments<R>(h);
  if (rho_out) __stcs(rho_out + x, (float)m.rho);
  if (u_out) {
    __stcs(u_out + x, (float)m.ux);
    __stcs(u_out + n + x, (float)m.uy);
    __stcs(u_out + 2 * n + x, (float)m.uz);
  }
  if (!wss_out) return;
  if (!wall) {
    __stcs(wss_out + x, __int_as_float(0x7fc00000));  // NaN
    return;
  }
  R nx = 0, ny = 0, nz = 0;
  if (normal) {
    nx = R(normal[x]);
    ny = R(normal[n + x]);
    nz = R(normal[2 * n + x]);
  } else {
    // fallback normal: the sum of c_j over the pull directions across a wall
    int sx = 0, sy = 0, sz = 0;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const int b = (wall >> (i - 1)) & 1;
      sx += cx(i) * b;
      sy += cy(i) * b;
      sz += cz(i) * b;
    }
    nx = R(sx);
    ny = R(sy);
    nz = R(sz);
    R l = sqrt(nx * nx + ny * ny + nz * nz);
    nx /= l; ny /= l; nz /= l;
  }
  R usq15 = R(1.5) * (m.ux * m.ux + m.uy * m.uy + m.uz * m.uz);
  R pxx = 0, pyy = 0, pzz = 0, pxy = 0, pxz = 0, pyz = 0;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    // only the components that c_i has: a product with 0 is not optimised
    // away, and in FP64 the zero terms were half of the kernel's arithmetic
    const R d = h[i] - heq<R>(i, m.drho, m.rho, m.ux, m.uy, m.uz, usq15);
    if (cx(i)) pxx += d;
    if (cy(i)) pyy += d;
    if (cz(i)) pzz += d;
    if (cx(i) && cy(i)) pxy = cx(i) * cy(i) > 0 ? pxy + d : pxy - d;
    if (cx(i) && cz(i)) pxz = cx(i) * cz(i) > 0 ? pxz + d : pxz - d;
    if (cy(i) && cz(i)) pyz = cy(i) * cz(i) > 0 ? pyz + d : pyz - d;
  }
  R k = -(R(1) - R(0.5) * omega_of<R>(p));
  R tx = k * (pxx * nx + pxy * ny + pxz * nz);
  R ty = k * (pxy * nx + pyy * ny + pyz * nz);
  R tz = k * (pxz * nx + pyz * ny + pzz * nz);
  R tn = tx * nx + ty * ny + tz * nz;
  tx -= tn * nx;
  ty -= tn * ny;
  tz -= tn * nz;
  __stcs(wss_out + x, (float)sqrt(tx * tx + ty * ty + tz * tz));
}

// Shifted pre-collision state f(t) - w into out [19][n] (row < 0), or only
// direction `row` into out [n].
template <typename S, int MODE, bool CT>
__global__ void __launch_bounds__(READ) k_state(const S* __restrict__ fin, const IndexTables ix,
                                                const LinkRec* __restrict__ links, const double* __restrict__ amp,
                                                const StepParams p, S* __restrict__ out, int row) {
  using R = typename Real<S>::type;
  const int64_t n = p.n;
  const int64_t x = (int64_t)blockIdx.x * READ + threadIdx.x;
  if (x >= n) return;
  if (MODE == 2 && row >= 0) {  // one direction of the AA gather: its own slot only
    const int32_t s = row ? ix.src[(int64_t)(row - 1) * p.sn + x] : -1;
    out[x] = fin[s >= 0 ? (int64_t)lane_opp(row) * n + s : (int64_t)row * n + x];
    return;
  }
  R h[Q];
  load_state<S, MODE, CT, false>(fin, ix, links, amp, p, x, (uint32_t)(x / CT_TILE), h);
  if (row >= 0) {
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (i == row) out[x] = from_real<S>(h[i]);
    return;
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) stpop<S>(out + (int64_t)i * n + x, h[i]);
}

// f = f^eq(rho0, u0) (Section 3.1 step 1), stored shifted.
template <typename S>
__global__ void __launch_bounds__(BLOCK) k_init(S* __restrict__ f, int64_t n, double rho0,
                                                const float* __restrict__ u0) {
  using R = typename Real<S>::type;
  const int64_t x = (int64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (x >= n) return;
  R ux = 0, uy = 0, uz = 0;
  if (u0) {
    ux = R(u0[x]);
    uy = R(u0[n + x]);
    uz = R(u0[2 * n + x]);
  }
  R drho = R(rho0 - 1.0);
  R usq15 = R(1.5) * (ux * ux + uy * uy + uz * uz);
#pragma unroll
  for (int i = 0; i < Q; ++i) f[(int64_t)i * n + x] = from_real<S>(heq<R>(i, drho, R(1) + drho, ux, uy, uz, usq15));
}

// ---------------------------------------------------------------------------
// FP64 reductions.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double r = 0;
  if (threadIdx.x == 0)
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) r += sh[k];
  __syncthreads();
  return r;  // valid in thread 0
}

// The sums of a state in two launches.  k_sums: blocks [0, nmass) write the
// sums of drho (mass - sites) over `per` x 256 sites of [lo, hi) each into
// part[block]; in the A-B scheme the blocks after them take 256 link records
// each and write the mass that each link lets in, recomputed from the
// post-collision state s'(t-1), into lflux (the AA steps record it there
// themselves).  With MON the last blocks take 256 entries of the iolets' site
// lists each and write |u|^2 and rho of f(t) into msite.  k_sums_finish adds
// them up in a fixed order.  One thread a link or site, whatever the number
// of iolets: one block an iolet walked thousands of links in a chain of
// dependent loads (26 us for 2 iolets of 2,000 links; now a few).
template <typename S, int MODE, bool CT, bool MON>
__global__ void __launch_bounds__(BLOCK) k_sums(const S* __restrict__ fin, const IndexTables ix,
                                                const LinkRec* __restrict__ links, const double* __restrict__ amp,
                                                const StepParams p, int64_t lo, int64_t hi, int per, unsigned nmass,
                                                unsigned nflux, int64_t nlinks, int64_t nlist,
                                                const int32_t* __restrict__ ilist, double* __restrict__ part,
                                                double* __restrict__ lflux, double* __restrict__ msite) {
  using R = typename Real<S>::type;
  const int64_t n = p.n;
  pdl_trigger();  // k_sums_finish waits for this kernel's end
  if (blockIdx.x < nmass) {
    __shared__ double sh[BLOCK / 32];
    const int64_t x0 = lo + (int64_t)blockIdx.x * (per * BLOCK) + threadIdx.x;
    const int count = x0 >= hi ? 0 : (int)min((int64_t)per, (hi - x0 + BLOCK - 1) / BLOCK);
    const double d = mass_sum<R>(count, [&](int k, R* h) {
      const int64_t x = x0 + k * BLOCK;
      load_state<S, MODE, CT, false>(fin, ix, links, amp, p, x, (uint32_t)(x / CT_TILE), h);
    });
    const double s = block_sum(d, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    return;
  }
  if (blockIdx.x < nmass + nflux) {
    const int64_t r = (int64_t)(blockIdx.x - nmass) * BLOCK + threadIdx.x;
    if (r >= nlinks) return;
    const LinkRec L = links[r];
    const int64_t x = L.site;
    R own[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) own[i] = ldpop(fin + (int64_t)i * n + x);
    const Macro<R> ms = moments<R>(own);
    const int j = L.dir;
    R out = R(0);
#pragma unroll
    for (int i = 1; i < Q; ++i)
      if (i == opp(j)) out = own[i];
    R val = R(0);
#pragma unroll
    for (int i = 1; i < Q; ++i)
      if (i == j) val = iolet_value<R>(i, L, out, ms.rho, ms.ux, ms.uy, ms.uz, amp, p);
    lflux[r] = (double)val - (double)out;
    return;
  }
  if (MON) {
    const int64_t q = (int64_t)(blockIdx.x - nmass - nflux) * BLOCK + threadIdx.x;
    if (q >= nlist) return;
    const int64_t x = ilist[q];
    R h[Q];
    load_state<S, MODE, false, false>(fin, ix, links, amp, p, x, 0u, h);
    const Macro<R> m = moments<R>(h);
    msite[2 * q] = (double)m.ux * m.ux + (double)m.uy * m.uy + (double)m.uz * m.uz;
    msite[2 * q + 1] = (double)m.rho;
  }
}

// Final sums, a block each, in a fixed order: block 0, out[0] = n + the mass
// partials; blocks 1 .. K, out[1 + k] = flux of iolet k, the sum over its link
// records (0 when the state did not come from a step); then, for the monitor,
// mon[k] = max |u| and mon[K + k] = mean rho over the sites linked to iolet k.
__global__ void __launch_bounds__(512) k_sums_finish(const double* __restrict__ part, int64_t nb, int64_t n, int K,
                                                     const double* __restrict__ lflux,
                                                     const int64_t* __restrict__ begin, int have_flux,
                                                     const double* __restrict__ msite,
                                                     const int64_t* __restrict__ ioff, double* __restrict__ out,
                                                     double* __restrict__ mon) {
  __shared__ double sh[512 / 32];
  const int b = blockIdx.x;
  pdl_wait();
  if (b <= K) {
    const double* v = b == 0 ? part : lflux;
    const int64_t lo = b == 0 ? 0 : begin[b - 1], hi = b == 0 ? nb : (have_flux ? begin[b] : begin[b - 1]);
    double acc = 0;
#pragma unroll 4
    for (int64_t r = lo + threadIdx.x; r < hi; r += 512) acc += v[r];
    const double s = block_sum(acc, sh);
    if (threadIdx.x == 0) out[b] = b == 0 ? (double)n + s : s;
    return;
  }
  const int k = b - K - 1;
  const int64_t lo = ioff[k], hi = ioff[k + 1];
  double umax = 0, rsum = 0;
#pragma unroll 4
  for (int64_t q = lo + threadIdx.x; q < hi; q += 512) {
    umax = fmax(umax, sqrt(msite[2 * q]));
    rsum += msite[2 * q + 1];
  }
  const double rs = block_sum(rsum, sh);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) umax = fmax(umax, __shfl_down_sync(FULL_MASK, umax, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = umax;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 512 / 32; ++w) umax = fmax(umax, sh[w]);
    mon[k] = umax;
    mon[K + k] = hi > lo ? rs / (double)(hi - lo) : 0.0;
  }
}

// ---------------------------------------------------------------------------
// dispatch
// ---------------------------------------------------------------------------
template <template <typename> class F, typename... A>
cudaError_t dispatch(int precision, A... a) {
  switch (precision) {
    case HLB_FP32: return F<float>::run(a...);
    case HLB_BF16: return F<__nv_bfloat16>::run(a...);
    case HLB_FP16: return F<__half>::run(a...);
    case HLB_FP64: return F<double>::run(a...);
  }
  return cudaErrorInvalidValue;
}

inline unsigned iolet_blocks(const hlb_solver* h, int threads) {
  return (unsigned)((h->n_iolet_sites * kStepIoletLanes + threads - 1) / threads);
}
// Prefetch distance of the two-site kernels, in tiles.  An FP32 state that stays
// in L2 has nothing to fetch ahead, and the hints for its rows only cost: none
// below 600k sites.
inline uint32_t prefetch_form(const hlb_solver* h) { return h->offset_major ? kPrefetchOffsets : 0u; }
template <typename S>
uint32_t pair_prefetch(const hlb_solver* h) {
  return sizeof(S) == 4 && h->n < 600000 ? 0u : (uint32_t)h->n_sm * 3u;
}
// Whether the offset-form tiles of k_step2 (1 to 14 % of a vessel lattice's) take
// two sites a thread.  us a step, one site after the other / at once: FP32 100k
// sites 4.28 / 4.97, 150k 5.18 / 5.22, 196k 5.68 / 5.41, 250k 7.08 / 6.52, 600k
// 16.1 / 14.9; BF16 100k 4.13 / 4.03, 150k 4.74 / 5.29, 196k 5.17 / 5.31, 250k
// 6.27 / 5.90, 600k 11.0 / 10.5.  Below about a wave of blocks what differs is the
// trigger: at once, a tile lets the next step's blocks in as soon as it starts,
// and they settle unevenly on the SMs beside it.
template <typename S>
bool pair_tiles(const hlb_solver* h) {
  return h->offset_major || h->n >= (sizeof(S) == 4 ? 175000 : 225000);
}
// 16-bit AA odd steps of fewer sites take one site a thread: the shorter thread
// is done sooner.  BF16, one site / two: 300k sites 9.92 / 10.08 us, 400k 10.95 /
// 11.01, 600k 13.9 / 13.7.
constexpr int64_t kOddPairSites = 450000;
// FP32 AA steps of fewer sites take two sites a thread in offset form too, their
// iolet sites in the grid: (x, y, z) order 50k sites 4.1 us against 5.5 (one site
// a thread and the pass), 500k 13.5 / 15.3, 2.0M 62.5 / 59.8, 8.0M 245 / 224.
constexpr int64_t kOffsetPairSites = 1000000;
constexpr int64_t kSpreadSites = 4000000;
inline uint32_t spread_factor(uint32_t iolet, uint32_t blocks) {
  return blocks ? (uint32_t)((((uint64_t)iolet << 32) + blocks - 1) / blocks) : 0u;
}
// The grid of a whole step with bulk blocks of `sites` sites and `threads`
// threads, its iolet blocks among those of their own sites.  A segment's iolet
// blocks are fewer than its blocks (its last holds the ones left over), so
// spread_factor stays below 2^32.
unsigned spread_iolets(const hlb_solver* h, int sites, int threads, IoletSpread* sp) {
  const int per = threads / kStepIoletLanes;
  const uint32_t bulk = (uint32_t)((h->n + sites - 1) / sites), all = iolet_blocks(h, threads);
  sp->segments = kSpread;
  for (int s = 0; s <= kSpread; ++s) {
    const int64_t x = s * h->spread_sites;
    const bool end = x >= h->n;
    sp->io[s] = end ? all : (uint32_t)(h->spread_count[(size_t)s] / per);
    sp->blk[s] = (end ? bulk : (uint32_t)(x / sites)) + sp->io[s];
  }
  for (int s = 0; s < kSpread; ++s) sp->k[s] = spread_factor(sp->io[s + 1] - sp->io[s], sp->blk[s + 1] - sp->blk[s]);
  return bulk + all;
}
// `bulk` bulk blocks with `iolet` iolet blocks spread evenly among them.  Iolet
// blocks alone get one bulk block, which has nothing to do (kNoTile).
unsigned spread_evenly(uint32_t bulk, uint32_t iolet, IoletSpread* sp) {
  if (bulk == 0 && iolet > 0) bulk = 1;
  sp->segments = 1;
  sp->blk[0] = sp->io[0] = 0;
  sp->k[0] = spread_factor(iolet, bulk + iolet);
  return bulk + iolet;
}

// One pull A-B gather step over the bulk tiles [tile0, tile0 + ntiles) and,
// with `iolets`, the iolet sites (the whole step: tile0 = 0, all tiles).
template <typename S>
cudaError_t launch_gather(const hlb_solver* h, const void* fin, void* fout, const StepParams& p, uint32_t tile0,
                          uint32_t ntiles, bool iolets, cudaStream_t s) {
  // a whole step past L2: the iolet blocks beside their sites (FP32 8.0M sites 215 -> 204 us, 20M 497 -> 483;
  // 16 bits the same); a small lattice, or a part of the step: evenly among its tiles, which needs no search
  // (0.5M sites, BF16: 10.0 us a step, 10.5 with it)
  const bool whole = iolets && tile0 == 0 && ntiles == grid_for(h->n) && (h->n >= kSpreadSites || sizeof(S) == 8);
  IoletSpread spread;
  if (ntiles == 0) tile0 = kNoTile;
  if constexpr (sizeof(S) <= 4) {
    if (h->compact) {
      const unsigned grid = whole ? spread_iolets(h, CT_TILE, PAIR, &spread)
                                  : spread_evenly(ntiles, iolets ? iolet_blocks(h, PAIR) : 0u, &spread);
      if (grid == 0) return cudaSuccess;
      auto kernel = pair_tiles<S>(h) ? (h->off32 ? k_step2<S, false, true> : k_step2<S, true, true>)
                                     : (h->off32 ? k_step2<S, false, false> : k_step2<S, true, false>);
      return launch_pdl(kernel, grid, PAIR, s, (const S*)fin, (S*)fout, h->index(),
                        h->d_links, h->d_amp, h->d_iolet_sites, h->n_iolet_sites, spread,
                        pair_prefetch<S>(h) ? pair_prefetch<S>(h) | prefetch_form(h) : 0u, tile0, p);
    }
  }
  const unsigned grid = whole ? spread_iolets(h, BLOCK, BLOCK, &spread)
                              : spread_evenly(ntiles, iolets ? iolet_blocks(h, BLOCK) : 0u, &spread);
  if (grid == 0) return cudaSuccess;
  constexpr bool CT = sizeof(S) > 4;  // FP64 only: the others take two sites a thread
  auto kernel = h->compact ? (h->off32 ? k_step<S, false, CT> : k_step<S, true, CT>)
                           : (h->off32 ? k_step<S, false, false> : k_step<S, true, false>);
  return launch_pdl(kernel, grid, BLOCK, s, (const S*)fin, (S*)fout, h->index(), h->d_links, h->d_amp,
                    h->d_iolet_sites, h->n_iolet_sites, spread, (uint32_t)h->n_sm * 5u | prefetch_form(h), tile0, p);
}

template <typename S>
struct StepOp {
  static cudaError_t run(const hlb_solver* h, const void* fin, void* fout, bool gather, int64_t tb,
                         cudaStream_t s) {
    StepParams p = h->params(tb);
    if (gather) return launch_gather<S>(h, fin, fout, p, 0, grid_for(h->n), true, s);
    return launch_pdl(k_step_local<S>, grid_for(h->n), BLOCK, s, (const S*)fin, (S*)fout, p);
  }
};

template <typename S>
struct StepRangeOp {
  static cudaError_t run(const hlb_solver* h, const void* fin, void* fout, int64_t tb, int64_t tile0,
                         int64_t ntiles, bool iolets, cudaStream_t s) {
    StepParams p = h->params(tb);
    return launch_gather<S>(h, fin, fout, p, (uint32_t)tile0, (uint32_t)ntiles, iolets, s);
  }
};

// Whether an AA step takes its iolet sites in its own grid or leaves them to
// k_aa_fix.  In the grid they save a launch and its wait, but hold slots of the
// bulk blocks while they wait for scattered loads.  Measured per step, in the
// grid against the pass, FP32: 0.5M sites 13.0 / 15.1 us, 1.0M 23.6 / 26.4, 2.0M
// 54.9 / 57.8, 8.0M 214 / 210, 20M 503 / 492.  16-bit storage gains less (2.0M
// 38.6 / 38.2, 20M 345 / 312) and keeps the pass, as FP64 and the int32 table do.
template <typename S>
bool aa_in_grid(const hlb_solver* h) {
  return sizeof(S) == 4 && h->compact && h->n < (h->offset_major ? kOffsetPairSites : 4000000);
}

// The iolet blocks of a grid with `bulk` bulk blocks of `threads` threads.
template <bool GRID>
AAIolets aa_iolets(const hlb_solver* h, unsigned bulk, int threads) {
  const unsigned gi = GRID ? iolet_blocks(h, threads) : 0u;
  return {h->d_icode, h->d_links, h->d_amp, h->d_iolet_sites, h->n_iolet_sites, h->d_imask, h->d_lflux, gi,
          make_block_div(gi ? (bulk + gi) / gi : 1)};
}

template <typename S, bool GRID>
cudaError_t launch_aa(const hlb_solver* h, S* A, bool odd, const StepParams& p, cudaStream_t s) {
  const unsigned g = grid_for(h->n);
  if (odd) {
    if constexpr (sizeof(S) <= 4) {
      if (h->compact && (sizeof(S) == 4 ? !h->offset_major || h->n < kOffsetPairSites
                                        : !h->offset_major && h->n >= kOddPairSites)) {
        const AAIolets io = aa_iolets<GRID>(h, g, PAIR);
        return launch_pdl(h->off32 ? k_aa_odd2<S, false, GRID> : k_aa_odd2<S, true, GRID>, g + io.blocks, PAIR, s, A,
                          h->index(), io, h->offset_major ? 0u : pair_prefetch<S>(h), p);
      }
    }
    if constexpr (!GRID) {
      return launch_pdl(h->compact ? (h->off32 ? k_aa_odd<S, false, true> : k_aa_odd<S, true, true>)
                                   : (h->off32 ? k_aa_odd<S, false, false> : k_aa_odd<S, true, false>),
                        g, BLOCK, s, A, h->index(), (uint32_t)h->n_sm * (h->off32 ? 3u : 4u) | prefetch_form(h), p);
    }
    return cudaErrorInvalidValue;  // GRID: compact FP32
  }
  if constexpr (sizeof(S) == 2) {
    if (h->n % 2 == 0) return launch_pdl(k_aa_even2<S>, grid_for(h->n / 2), BLOCK, s, A, p);
  }
  const AAIolets io = aa_iolets<GRID>(h, g, BLOCK);
  return launch_pdl(k_aa_even<S, GRID>, g + io.blocks, BLOCK, s, A, io, p);
}

template <typename S>
struct AAOp {
  static cudaError_t run(const hlb_solver* h, void* A, bool odd, int64_t t, cudaStream_t s) {
    const StepParams p = h->params(t);
    if constexpr (sizeof(S) == 4) {
      if (aa_in_grid<S>(h)) return launch_aa<S, true>(h, (S*)A, odd, p, s);
    }
    const cudaError_t e = launch_aa<S, false>(h, (S*)A, odd, p, s);
    if (e != cudaSuccess || h->n_iolet_sites == 0) return e;
    constexpr int per_block = 256 / kFixLanes;  // iolet sites a block
    const unsigned g = (unsigned)((h->n_iolet_sites + per_block - 1) / per_block);
    return launch_pdl(odd ? k_aa_fix<S, true> : k_aa_fix<S, false>, g, 256, s, (S*)A, h->d_icode, h->d_links,
                      h->d_amp, h->d_iolet_sites, h->n_iolet_sites, p, h->d_lflux);
  }
};

#define HLB_MODE_SWITCH(mode, KERNEL_LAUNCH)                  \
  switch (mode) {                                              \
    case HLB_READ_GATHER_AB: { constexpr int M = HLB_READ_GATHER_AB; KERNEL_LAUNCH; break; } \
    case HLB_READ_GATHER_AA: { constexpr int M = HLB_READ_GATHER_AA; KERNEL_LAUNCH; break; } \
    default: { constexpr int M = HLB_READ_LOCAL; KERNEL_LAUNCH; break; }                      \
  }

template <typename S>
struct MacroOp {
  static cudaError_t run(const hlb_solver* h, const void* fin, int mode, int64_t tb, float* rho, float* u,
                         float* wss, cudaStream_t s) {
    StepParams p = h->params(tb);
    const float* nrm = h->has_normals ? h->d_normal : nullptr;
    const unsigned g = (unsigned)((h->n + READ - 1) / READ);
    HLB_MODE_SWITCH(mode, ((h->compact ? k_macros<S, M, true> : k_macros<S, M, false>)<<<g, READ, 0, s>>>(
                              (const S*)fin, h->index(), h->d_links, h->d_amp, nrm, p, rho, u, wss)));
    return cudaGetLastError();
  }
};

// Windkessel outlets after a step (block k = iolet k; other iolets return).
// q = -(mass that enters through outlet k to produce the current state f):
//  * AA: the fix-up pass has just written f's boundary values with ioval[k]
//    and recorded the per-link masses; q is their sum.
//  * A-B: f's boundary values are applied by the next gather.  That gather
//    uses the value computed one update earlier (iovnext[k]), which `shift`
//    moves into ioval[k]; q is then recomputed from the post-collision state
//    `fin` with it, exactly as the gather will see it.
// Then rho_c <- rho_c + (q - (rho_c - rho_d) / Rd) / C and the next ghost
// density rho_c + Rp q (C = 0: rho_d + (Rp + Rd) q) goes to ioval[k] (AA) or
// iovnext[k] (A-B), minus 1.
template <typename S, bool AA>
__global__ void __launch_bounds__(BLOCK) k_wk_update(const S* __restrict__ fin, const LinkRec* __restrict__ links,
                                                     const double* __restrict__ amp, const StepParams p,
                                                     const int64_t* __restrict__ begin,
                                                     const double* __restrict__ lflux,
                                                     const double* __restrict__ par, double* __restrict__ state,
                                                     double* ioval, double* __restrict__ iovnext, int shift) {
  using R = typename Real<S>::type;
  // Links between two block barriers (pull).  50k sites with outlets, single steps:
  // FP32 10.8 us at one a thread, 10.6 at two and four; FP64 42 us at one and two, 50
  // to 70 at four (8 KB: it lasts as long as the SM that gets most blocks).
  constexpr int CHUNK = AA ? 1 : 2 * BLOCK;
  __shared__ double sh[BLOCK / 32], mass[CHUNK];
  const int k = blockIdx.x;
  pdl_wait();
  pdl_trigger();
  if (!((p.coupled[k >> 6] >> (k & 63)) & 1ull)) return;  // uniform per block
  if (!AA && shift) {
    if (threadIdx.x == 0) ioval[k] = iovnext[k];
    __syncthreads();  // io_val(p, k) below reads it (p.ioval == ioval)
  }
  const int64_t n = p.n;
  double acc = 0;
  if (AA)  // no multi-step launches, so no order to keep to: all threads add
    for (int64_t r = begin[k] + threadIdx.x; r < begin[k + 1]; r += BLOCK) acc += lflux[r];
  for (int64_t r0 = begin[k], end = AA ? r0 : begin[k + 1]; r0 < end; r0 += CHUNK) {
    const int count = (int)min((int64_t)CHUNK, end - r0);
    for (int m = threadIdx.x; m < count; m += BLOCK) {
      const int64_t r = r0 + m;
      const LinkRec L = links[r];
      const int64_t x = L.site;
      R own[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) own[i] = ldpop(fin + (int64_t)i * n + x);
      const Macro<R> ms = moments<R>(own);
      const R out = ldpop(fin + (int64_t)lane_opp(L.dir) * n + x);
      const R a = BC<R>::amp(p, amp, L.kind == 0 && L.group >= 0 ? L.group : 0);
      const R val = lane_iolet_value<R>(L.dir, L, out, ms.rho, ms.ux, ms.uy, ms.uz, a, BC<R>::val(p, L.iolet), p);
      mass[m] = (double)val - (double)out;
    }
    // in the order of a multi-step launch's outlet blocks (hlb_multi.cu)
    __syncthreads();
    if (threadIdx.x < kWkLanes)
      for (int m = threadIdx.x; m < count; m += kWkLanes) acc += mass[m];
    if (r0 + CHUNK < end) __syncthreads();
  }
  const double flux = block_sum(acc, sh);
  if (threadIdx.x == 0) {
    const double Rp = par[4 * k], C = par[4 * k + 1], Rd = par[4 * k + 2], rho_d = par[4 * k + 3];
    const double q = -flux;
    double rho_c = state[2 * k];
    (AA ? ioval : iovnext)[k] = wk_advance(Rp, C, Rd, rho_d, q, &rho_c);
    state[2 * k] = rho_c;
    state[2 * k + 1] = q;
  }
}

// Windkessel outlets at initialisation: no outflow history.
__global__ void k_wk_reset(int32_t n_iolets, const StepParams p, const double* __restrict__ par,
                           double* __restrict__ state, double* __restrict__ ioval, double* __restrict__ iovnext) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_iolets || !((p.coupled[k >> 6] >> (k & 63)) & 1ull)) return;
  const double C = par[4 * k + 1], rho_d = par[4 * k + 3];
  if (!(C > 0)) state[2 * k] = rho_d;
  state[2 * k + 1] = 0.0;
  ioval[k] = iovnext[k] = state[2 * k] - 1.0;
}

template <typename S>
struct WkOp {
  static cudaError_t run(const hlb_solver* h, const void* fin, int64_t tb, bool shift, cudaStream_t s) {
    StepParams p = h->params(tb);
    const int64_t* begin = (const int64_t*)(h->d_red + hlb_reduce_partials(h->n));  // link ranges stored after the partials
    if (h->scheme == HLB_AA)
      return launch_pdl(k_wk_update<S, true>, (unsigned)h->n_iolets, BLOCK, s, (const S*)nullptr, h->d_links,
                        h->d_amp, p, begin, h->d_lflux, h->d_wkpar, h->d_wkstate, h->d_ioval, h->d_iovnext, 0);
    return launch_pdl(k_wk_update<S, false>, (unsigned)h->n_iolets, BLOCK, s, (const S*)fin, h->d_links, h->d_amp,
                      p, begin, (const double*)nullptr, h->d_wkpar, h->d_wkstate, h->d_ioval, h->d_iovnext,
                      shift ? 1 : 0);
  }
};

template <typename S>
struct StateOp {
  static cudaError_t run(const hlb_solver* h, const void* fin, int mode, int64_t tb, void* out, int row,
                         cudaStream_t s) {
    StepParams p = h->params(tb);
    const unsigned g = (unsigned)((h->n + READ - 1) / READ);
    HLB_MODE_SWITCH(mode, ((h->compact ? k_state<S, M, true> : k_state<S, M, false>)<<<g, READ, 0, s>>>(
                              (const S*)fin, h->index(), h->d_links, h->d_amp, p, (S*)out, row)));
    return cudaGetLastError();
  }
};

template <typename S>
struct InitOp {
  static cudaError_t run(const hlb_solver* h, void* f, double rho0, const float* u0, cudaStream_t s) {
    k_init<S><<<grid_for(h->n), BLOCK, 0, s>>>((S*)f, h->n, rho0, u0);
    return cudaGetLastError();
  }
};

template <typename S, int MODE, bool CT>
void launch_sums(const hlb_solver* h, const S* fin, const StepParams& p, bool mass, bool links, bool monitor, cudaStream_t s) {
  const int64_t lo = h->owned_lo, hi = h->owned_hi;
  const int per = mass_sites(h->n);
  const unsigned nmass = mass ? (unsigned)mass_blocks(hi - lo, per) : 0u, nflux = links ? grid_for(h->n_links) : 0u;
  const unsigned nmon = monitor ? grid_for(h->n_ilist) : 0u;
  if (nmass + nflux + nmon == 0) return;
  (monitor ? k_sums<S, MODE, CT, true> : k_sums<S, MODE, CT, false>)<<<nmass + nflux + nmon, BLOCK, 0, s>>>(
      fin, h->index(), h->d_links, h->d_amp, p, lo, hi, per, nmass, nflux, h->n_links, h->n_ilist, h->d_ilist, h->d_red,
      h->d_lflux, h->d_msite);
}

template <typename S>
struct ReduceOp {
  static cudaError_t run(const hlb_solver* h, const void* fin, int mode, int64_t tb, bool have_flux, bool totals,
                         bool monitor, double* out, cudaStream_t s) {
    StepParams p = h->params(tb);
    const int64_t owned = h->owned_hi - h->owned_lo;
    // the A-B scheme's fluxes are recomputed; the AA steps have recorded them
    const bool links = totals && have_flux && h->scheme != HLB_AA && h->n_links > 0;
    HLB_MODE_SWITCH(mode, (h->compact ? launch_sums<S, M, true>(h, (const S*)fin, p, totals, links, monitor, s)
                                      : launch_sums<S, M, false>(h, (const S*)fin, p, totals, links, monitor, s)));
    const int K = h->n_iolets;
    const int64_t* begin = (const int64_t*)(h->d_red + hlb_reduce_partials(h->n));  // link ranges stored after the partials
    if (const cudaError_t e = cudaGetLastError(); e != cudaSuccess) return e;
    // programmatic launch: its blocks are there when k_sums ends (monitor of 45k sites without fluxes 29 -> 27 us)
    return launch_pdl(
        k_sums_finish, (unsigned)(monitor ? 1 + 2 * K : 1 + K), 512, s, h->d_red, totals ? mass_blocks(owned, mass_sites(h->n)) : 0, owned, K, h->d_lflux, begin, totals && have_flux ? 1 : 0, h->d_msite, h->d_ioff, out, out + 1 + K);
  }
};

}  // namespace

int64_t hlb_reduce_partials(int64_t n) { return mass_blocks(n, mass_sites(n)); }

int64_t hlb_reduce_slots(int64_t n, int32_t n_iolets) {
  // per-block partials, iolet link ranges (int64, n_iolets + 1), final outputs: mass and
  // fluxes (1 + n_iolets), monitor (2 n_iolets), then the status word of the multi-step launches
  return hlb_reduce_partials(n) + (n_iolets + 1) + (1 + 3 * (int64_t)n_iolets) + 1;
}

cudaError_t hlb_launch_step(const hlb_solver* h, const void* fin, void* fout, bool gather, int64_t tb,
                            cudaStream_t s) {
  return dispatch<StepOp>(h->precision, h, fin, fout, gather, tb, s);
}
cudaError_t hlb_launch_step_range(const hlb_solver* h, const void* fin, void* fout, int64_t tb, int64_t tile0,
                                  int64_t ntiles, bool iolets, cudaStream_t s) {
  return dispatch<StepRangeOp>(h->precision, h, fin, fout, tb, tile0, ntiles, iolets, s);
}
cudaError_t hlb_launch_aa(const hlb_solver* h, void* A, bool odd, int64_t t, cudaStream_t s) {
  return dispatch<AAOp>(h->precision, h, A, odd, t, s);
}
cudaError_t hlb_launch_macros(const hlb_solver* h, const void* fin, int mode, int64_t tb, float* rho, float* u,
                              float* wss, cudaStream_t s) {
  return dispatch<MacroOp>(h->precision, h, fin, mode, tb, rho, u, wss, s);
}
cudaError_t hlb_launch_wk_update(const hlb_solver* h, const void* fin, int64_t tb, bool shift, cudaStream_t s) {
  return dispatch<WkOp>(h->precision, h, fin, tb, shift, s);
}
cudaError_t hlb_launch_wk_reset(const hlb_solver* h, cudaStream_t s) {
  StepParams p = h->params(h->t);
  k_wk_reset<<<(unsigned)((h->n_iolets + 127) / 128), 128, 0, s>>>(h->n_iolets, p, h->d_wkpar, h->d_wkstate,
                                                                   h->d_ioval, h->d_iovnext);
  return cudaGetLastError();
}
cudaError_t hlb_launch_state(const hlb_solver* h, const void* fin, int mode, int64_t tb, void* out, int row,
                             cudaStream_t s) {
  return dispatch<StateOp>(h->precision, h, fin, mode, tb, out, row, s);
}
cudaError_t hlb_launch_ctab(const hlb_solver* h, int32_t* misfit, cudaStream_t s) {
  const int64_t tiles = (h->sn + CT_TILE - 1) / CT_TILE;
  k_ctab_build<<<(unsigned)tiles, CT_TILE, 0, s>>>(h->d_src, h->n, h->sn, h->d_ctab, h->d_tbase, h->d_rtab,
                                                        h->d_rbase, misfit);
  return cudaGetLastError();
}
cudaError_t hlb_launch_init(const hlb_solver* h, void* f, double rho0, const float* u0, cudaStream_t s) {
  return dispatch<InitOp>(h->precision, h, f, rho0, u0, s);
}
cudaError_t hlb_launch_reduce(const hlb_solver* h, const void* fin, int mode, int64_t tb, bool have_flux, bool totals,
                              bool monitor, double* out_dev, cudaStream_t s) {
  return dispatch<ReduceOp>(h->precision, h, fin, mode, tb, have_flux, totals, monitor, out_dev, s);
}
