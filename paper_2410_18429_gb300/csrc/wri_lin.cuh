// Stencil passes over linear chunks of the x-y plane (complex64 and complex128).
//
// A work item is (system, chunk of L consecutive nodes of the x-y plane, z-chunk).  The planes of the
// input vectors stream through a ring of S shared-memory stages that one lane of a copy warp fills
// with untiled bulk copies (cp.async.bulk): the chunk plus nx nodes on either side, one contiguous
// piece of memory per plane and vector.  The y neighbours of node e are then e - nx and e + nx of the
// same stage, the x neighbours e - 1 and e + 1, and the z neighbours stay in the thread's registers.
//
// Why chunks and not x-y boxes:
//   * one contiguous copy per plane and vector streams faster than the rows of a 36 x 10 box (two vectors
//     in and two out, 148^3, 32 systems: 6440 against 6015 GB/s), although it brings 2 nx / L halo nodes
//     per node (2.2 reads from L2 per node at nx = 148 against 1.4);
//   * the chunks of a plane cover it without the idle lanes of ragged boxes (84^2 in 32 x 8 boxes: 20 %,
//     148^2: 11 %, 81^2: 29 %);
//   * any extent and parity of nx works: a copy starts at the 16-byte boundary below its first node and
//     the consumers index from the remainder.
//
// Stretched axes.  With the node factors s_x s_y s_z taken out of A,
//   (A u)_n = s_x s_y s_z [ (omega^2 m + a_x + a_y + a_z) u_n + sum over the six neighbours of alpha u ],
//   alpha = 1 / (s(half) s(node) h^2),  a = -(alpha_- + alpha_+),
// a fully stretched node takes about 37 multiply-adds instead of 72, and multiplying by s = 1 + i sigma / omega
// takes two.  The profile of the layer depends only on the distance into it, so one table of npml + 1
// entries (formed on the host in FP64) serves all axes and both faces.  Warps without a stretched or
// boundary node use the plain 7-point formula; the choice is made once per item.
//
// One pass per plane: when plane k arrives, a thread completes the stencil of plane k - 1 (the z + 1 term
// is its own new value), computes plane k's without the z + 1 term and hands the stage back, so S - 1
// planes stay in flight.
//
// What binds: the complex64 phases run at 5.3 TB/s of DRAM traffic (148^3 x 16) with 55 to 57 % of the issue slots
// used, 253 (phase 1) and 262 (phase 2) warp instructions per 64 nodes and plane; FP64 passes run the FP64 pipe at
// 87-89 % of its rate.  Chunks of 512 nodes (half the halo) are slower (148^3 x 32 45.8 -> 47.8 us per system and
// iteration, 276 x 276 x 180 x 4 173 -> 181), and so are stages beyond three (the plane streams alone 550 -> 749 us
// with six).
//
// All waits are bounded as in wri_tma.cuh: a time-out raises the CTA's abort flag and the launch's error
// flag, the consumers leave on a barrier-reduced copy of it, and the copy warp waits for its own copies.
#pragma once

#include <type_traits>

#include "wri_launch.h"
#include "wri_march_impl.cuh"
#include "wri_tma.cuh"

namespace wri {

struct LinSet {
  int* err;                    // set to 1 by a CTA whose copy wait timed out
  unsigned long long wait_ns;  // time limit of every wait (global timer, ns)
  int withhold;                // test hook, -1 = off (TmaSet::withhold)
  int off_b, off_m, stage;     // bytes of a stage: field a at 0, field b, model, end
  int gz;                      // gradient: planes of the largest z-chunk
};

// The layer table of an operator application travels with the kernel arguments (it has no workspace).
template <int MODE>
struct LinTab {};
template <>
struct LinTab<M_APPLY> {
  int n;  // entries
  double v[kLinInlineTab * kLayerTab];
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

__device__ __forceinline__ float fma_r(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_r(double a, double b, double c) { return __fma_rn(a, b, c); }
// acc + a b and a b (complex a), acc + s b (real s)
template <typename C>
__device__ __forceinline__ C cfma(C a, C b, C acc) {
  return mkc(fma_r(a.x, b.x, fma_r(-a.y, b.y, acc.x)), fma_r(a.x, b.y, fma_r(a.y, b.x, acc.y)));
}
template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
  return mkc(fma_r(a.x, b.x, -(a.y * b.y)), fma_r(a.x, b.y, a.y * b.x));
}
template <typename R, typename C>
__device__ __forceinline__ C rfma(R s, C b, C acc) {
  return mkc(fma_r(s, b.x, acc.x), fma_r(s, b.y, acc.y));
}
// (1 + i t) a
template <typename R, typename C>
__device__ __forceinline__ C smul(R t, C a) {
  return mkc(fma_r(-t, a.y, a.x), fma_r(t, a.x, a.y));
}

// Coefficients of one axis at one node: neighbour weights alpha_-, alpha_+, their negated sum, and the
// imaginary part of s.  zp: the weight of the + neighbour without the node's own 1/s (z axis).
template <typename R>
struct AxisCoef {
  cx<R> am, ap, a0;
  R im;
};

template <typename R, bool CONJ>
__device__ __forceinline__ cx<R> tab_c(const R* e, int k) {
  return mkc(e[k], CONJ ? -e[k + 1] : e[k + 1]);
}

// entry of node i: layer distance, which face; false for an unstretched node
__device__ __forceinline__ bool layer_at(int i, int n, int npml, int& d, bool& lo, bool& hi) {
  if (npml == 0) return false;
  lo = i <= npml;
  hi = i >= n - 1 - npml;
  d = lo ? npml - i : i - (n - 1 - npml);
  return lo || hi;
}

template <typename R, bool CONJ>
__device__ __forceinline__ AxisCoef<R> axis_coef(const R* tab, int i, int n, int npml, R ih2, cx<R>* zp = nullptr) {
  AxisCoef<R> c;
  int d;
  bool lo, hi;
  if (!layer_at(i, n, npml, d, lo, hi)) {
    c.am = c.ap = mkc(ih2, R(0));
    c.a0 = mkc(R(-2) * ih2, R(0));
    c.im = R(0);
    if (zp) *zp = c.ap;
    return c;
  }
  const R* e = tab + kLayerTab * d;
  const cx<R> near_ = tab_c<R, CONJ>(e, 0), far_ = tab_c<R, CONJ>(e, 2);
  c.im = CONJ ? -e[6] : e[6];
  c.am = lo ? far_ : near_;
  c.ap = hi ? far_ : near_;
  c.a0 = (lo && hi) ? R(-2) * far_ : tab_c<R, CONJ>(e, 4);  // a single interior node lies at both faces
  if (zp) *zp = tab_c<R, CONJ>(e, hi ? 10 : 8);
  return c;
}

// element e of a staged model chunk (complex64 passes have a float model, FP64 passes either)
template <typename R>
__device__ __forceinline__ R model_smem(const unsigned char* p, int m_double, int e) {
  if (sizeof(R) == 8 && m_double) return R(reinterpret_cast<const double*>(p)[e]);
  return sizeof(R) == 8 ? R(widen(reinterpret_cast<const float*>(p)[e])) : R(reinterpret_cast<const float*>(p)[e]);
}

// The system's scalars, run by the NT consumer threads of the CTA that finished its last item.  Phase 1 adds
// lambda^2 |p|^2 of the receivers; phase 2 moves the receiver residual (r2 -= alpha lambda p, with the p that
// phase 1 stored) and adds lambda P^T r2 to s.
// One reduction, no vector that this launch wrote but at the receivers: with the fences that leaves
// (148^3 x 1 system 79.7 -> 71.9 us per iteration, x 64 sources x 3 grids 2331 -> 2266; half of it from the
// receivers' bits, which cost the borehole's CTAs a global load per plane when rows of x held them).
template <typename R, typename OR, int MODE, int NT, typename SYNC>
__device__ void finalize_lin(const Batch& b, const GroupDev& G, SysDev* sd, int sl, double* red) {
  typedef cx<R> C;
  typedef cx<OR> OC;
  const int tid = threadIdx.x;
  const long long off = (long long)sl * G.n;
  double part = 0.0;  // sums of the items, in item order per thread
  if (MODE != M_RES) {
    const double* pp = b.partial + sd->part_off;
    for (int t = tid; t < G.ntiles; t += NT) part += __ldcg(pp + t);
  }
  const R lam = R(G.lambda);
  C* r2 = (C*)b.r2;
  const R step = MODE == M_P2 ? R(sd->alpha * (double)lam) : R(0);
  const C* p = (MODE == M_P1 || MODE == M_P2) ? (const C*)G.p[pslot(b, sd->iter)] + off : nullptr;
  if (!(MODE == M_SH && G.rmap)) {
    // A receiver is a few trips to the L2 that nothing else of its system is left to hide: the next index is loaded
    // a receiver ahead and p, s and r2 together (index, then p, then s: 81^3 with 2025 receivers x 1 system 49.8 ->
    // 44.1 us per iteration, x 9 137 -> 125).  Two receivers at a time gave 41.0 and 124, but the registers they
    // hold spill in the plane loops: 148^3 x 4 206 -> 214.
    int next = sd->rec_begin + tid < sd->rec_end ? b.rec_idx[sd->rec_begin + tid] : 0;
    for (int k = sd->rec_begin + tid; k < sd->rec_end; k += NT) {
      const int node = next;
      if (k + NT < sd->rec_end) next = b.rec_idx[k + NT];
      if (MODE == M_P1) {
        part += (double)lam * (double)lam * (double)abs2(ldcg_c(p + node));
      } else if (MODE == M_RES) {
        r2[k] = ((const C*)b.lamd)[k] - lam * ldcg_c((const C*)G.x + off + node);
      } else {
        OC* S = (OC*)G.s + off + node;
        const OC s_old = ldcg_c(S);
        C r = r2[k];
        if (MODE == M_P2) r2[k] = r = r - step * ldcg_c(p + node);
        // the stencil pass left receiver nodes out of its partial sums
        const OC sn = to_c(to_c(s_old, R(0)) + lam * r, OR(0));
        *S = sn;
        part += (double)abs2(sn);
      }
    }
  }
  const double tot = block_sum<NT, SYNC>(part, red);
  if (tid == 0) {
    if (MODE == M_P1) p1_scalars(b, sd, tot);
    if (MODE == M_P2) p2_scalars(b, sd, tot);
    if (MODE == M_SH) sh_scalars(b, sd, tot);
    sd->ticket = 0u;
  }
}

// R: arithmetic; OR: type of the stencil's output vector; MODE: M_APPLY, M_SH, M_RES, M_P1, M_P2 or M_GRAD; NC
// consumer threads of NPT nodes each; GV: phase 2 adds S^H r64 (gvec); PAIR: a thread's two nodes are adjacent
// (16-byte accesses: nx even and every pointer aligned), otherwise they lie NC apart; S stages; XO: warps outside
// the y layers have loops of their own.
template <typename R, typename OR, int MODE, bool CONJ, int NC, int NPT, bool PAIR, bool GV, int S, int MINB, bool XO>
__global__ void __launch_bounds__(NC + 32, MINB) k_lin(const __grid_constant__ Batch b, const __grid_constant__ LinSet T,
                                                         const __grid_constant__ LinTab<MODE> tab_in) {
  typedef cx<R> C;
  typedef cx<OR> OC;
  static_assert(!PAIR || (NPT == 2 && sizeof(R) == 4), "pairs of complex64");
  constexpr int L = NC * NPT;
  static_assert(L == kLinChunk, "the threads cover a chunk");
  constexpr bool HASB = (MODE == M_P1 || MODE == M_P2);
  constexpr bool NORM = (MODE == M_P1 || MODE == M_P2 || MODE == M_SH);
  constexpr int NCW = NC / 32;
  constexpr bool GRAD = MODE == M_GRAD;
  // The stencil is formed from differences to the node, which are exact or nearly so for a resolved field, so
  // that the rounding of a coefficient acts on a difference.  complex128 takes an unstretched axis as the sum of
  // its two neighbours minus 2 u (fewer FP64 instructions), and x and y together as four minus 4 u where both are.
  // Its root mean square error is 1.8 units (2^-53 u / h^2) off the layers, 2.9 at a source, 5.4 where one axis is
  // stretched and 12.9 where all are (damped outgoing waves, 864 on four grids; z-march kernels 1.9, 3.2, 6.1, 16.3).
  // Cheaper forms lose: five neighbours in one sum saves 2 FP64 instructions of 19 off the layers (A^H on 81^3 x 9
  // 305 -> 297 us) but has 2.3 units there and 3.4 at a source, and the diagonal in one coefficient saves 4 of 19 to
  // 8 of 37 (264 us) at up to four times the error.
  constexpr bool DIFF = sizeof(R) == 4;
  // complex64: the first step of an item finishes a plane below it all the same (no check in the loop) and
  // its result is overwritten; complex128 saves the FP64 instructions
  constexpr bool DUMMY = sizeof(R) == 4;
  constexpr int CB = sizeof(C);
  constexpr int RS = PAIR ? 1 : NC;  // distance of a thread's nodes
  typedef FirstThreadsSync<NC> CSync;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ double red[NCW];
  __shared__ int s_last;
  __shared__ volatile int s_abort;
  __shared__ R s_tab[MODE == M_APPLY ? kLinInlineTab * kLayerTab : 1];
  unsigned char* smem = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
  const int SB = T.stage;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)S * SB);
  uint64_t* empty = full + S;
  double* gacc = reinterpret_cast<double*>(empty + S);  // gradient: [planes of the z-chunk][L]
  const int tid = threadIdx.x;
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], NCW);
    }
    mbar_init_done();
    s_abort = 0;
  }
  if constexpr (MODE == M_APPLY)
    for (int e = tid; e < tab_in.n * kLayerTab; e += NC + 32) s_tab[e] = R(tab_in.v[e]);
  __syncthreads();  // the only CTA-wide barrier: the copy warp leaves the consumers' barriers after it

  // what the item does; the same decision in both roles
  auto skip_item = [&](const SysDev* sd) -> bool {
    if (MODE == M_P1 || MODE == M_P2) return sd->state != ST_ACTIVE;
    if ((MODE == M_SH || MODE == M_RES) && (b.flavor == SH_REFINE || b.flavor == SH_PLAIN)) return sd->outer_done != 0;
    return false;
  };
  // the fields of F = a + coef b: at iteration 0 there is no older direction, b = a with coef 0
  auto field_a = [&](const GroupDev& G, int iter) -> const char* {
    return (const char*)(MODE == M_P1 ? G.s : MODE == M_P2 ? G.r1[iter & 1] : MODE == M_SH ? G.r1[0] : G.x);
  };
  auto field_b = [&](const GroupDev& G, int iter) -> const char* {
    return (const char*)(MODE == M_P2 ? G.t1 : iter > 0 ? G.p[pslot(b, iter - 1)] : G.s);
  };

  // ================================================================ copy warp
  if (tid >= NC) {
    if (tid != NC) return;
    // a copy wait of an earlier launch of this solve timed out: this launch copies nothing, and its consumers
    // find the flag in their first wait
    if (T.err && *(volatile const int*)T.err != 0) {
      s_abort = 1;
      return;
    }
    unsigned fills = 0;
    int st = 0;
    uint32_t par = 1;  // parity of the stage's previous release (first use: none)
    bool stop = false;
    for (long long item = blockIdx.x; item < b.nitems && !stop; item += gridDim.x) {
      const int gi = find_group(b, item);
      const GroupDev& G = b.g[gi];
      int sl = 0, tile = (int)(item - G.item0);
      if (!GRAD) item_coords32(b, G, item - G.item0, sl, tile);
      const SysDev* sd = (MODE == M_APPLY) ? nullptr : b.sys + (G.sys0 + sl);
      if (MODE != M_APPLY && skip_item(sd)) continue;
      const int plane = G.nx * G.ny;
      const int z0 = (tile % G.zsplit) * G.zc, z1 = min(z0 + G.zc, G.nz);
      const int c0 = (tile / G.zsplit) * G.chunk, c1 = min(c0 + G.chunk, plane);
      const int lo = max(c0 - G.nx, 0), hi = min(c1 + G.nx, plane);
      const int iter = HASB ? sd->iter : 0;
      const char* fa = field_a(G, iter) + (long long)sl * G.n * CB;
      const char* fb = HASB ? field_b(G, iter) + (long long)sl * G.n * CB : nullptr;
      const int em = G.m_double ? 8 : 4;
      // the gradient streams its z-chunk of one system after the other
      const int passes = GRAD ? G.nsys : 1;
      // Running addresses of the chunk's first node (plane k), and what an inner plane adds on either side.  A
      // copy starts at the 16-byte boundary below its first node and ends at the one above its last; node
      // c0 - nx lands (its address & 15) bytes into the region (always 0 where rows are whole 16-byte units).
      constexpr bool ALIGNED = PAIR || CB == 16;
      const int k0 = max(z0 - 1, 0);
      const long long fstep = (long long)plane * CB, mstep = (long long)plane * em;
      const uint32_t below = (uint32_t)(c0 - lo) * CB, above = (uint32_t)(hi - c1) * CB, mid = (uint32_t)(c1 - c0) * CB;
      const uint32_t halo = (uint32_t)G.nx * CB;  // bytes between the region's start and the chunk's
      uint64_t* const bars = full;
      auto copy = [&](uint32_t region, uintptr_t at, bool inner, int stage, bool issue) -> uint32_t {
        const uint32_t back = inner ? below : 0u;
        const uintptr_t first = at - back;
        const uint32_t pre = ALIGNED ? 0u : (uint32_t)(first & 15);
        const uint32_t len = mid + (inner ? below + above : 0u);
        const uint32_t bytes = ALIGNED ? len : (pre + len + 15) & ~15u;
        if (issue)
          bulk_load(region + (halo - back) + (ALIGNED ? 0u : (uint32_t)((at - halo) & 15) - pre), (const void*)(first - pre),
                    bytes, &bars[stage]);
        return bytes;
      };
      for (int pass = 0; pass < passes && !stop; ++pass) {
        uintptr_t pa = (uintptr_t)fa + ((long long)(GRAD ? pass : 0) * G.n + (long long)k0 * plane + c0) * CB;
        uintptr_t pb = HASB ? (uintptr_t)fb + ((long long)k0 * plane + c0) * CB : 0;
        uintptr_t pm = (uintptr_t)G.m + ((long long)k0 * plane + c0) * em;
        for (int k = k0; k <= min(z1, G.nz - 1); ++k, ++fills, pa += fstep, pb += fstep, pm += mstep) {
          if (fills >= (unsigned)S && !mbar_try_wait(&empty[st], par) &&
              !mbar_wait_or_abort(&empty[st], par, &s_abort, T.wait_ns)) {
            s_abort = 1;
            if (T.err) atomicExch(T.err, 1);
            stop = true;
            break;
          }
          // test hook (off unless the caller asks): this fill is never issued, so its "full" barrier
          // never completes and the consumers' bounded wait for it runs out
          if (!(blockIdx.x == 0 && (int)fills == T.withhold)) {
            const uint32_t base = smem_addr(smem) + (uint32_t)st * SB;
            const bool inner = k >= z0 && k < z1;  // the planes next to the z-chunk give z neighbours only
            const uint32_t mpre = (uint32_t)(pm & 15), mbytes = (mpre + (uint32_t)(c1 - c0) * em + 15) & ~15u;
            const uint32_t ba = copy(base, pa, inner, st, false);
            const uint32_t bb = !HASB ? 0u : ALIGNED ? ba : copy(base, pb, inner, st, false);
            mbar_expect_tx(&full[st], ba + bb + (inner ? mbytes : 0u));
            copy(base, pa, inner, st, true);
            if (HASB) copy(base + T.off_b, pb, inner, st, true);
            if (inner) bulk_load(base + T.off_m, (const void*)(pm - mpre), mbytes, &full[st]);
          }
          if (++st == S) {
            st = 0;
            par ^= 1;
          }
        }
      }
    }
    drain_copies<S>(full, fills, T.withhold);
    return;
  }

  // ================================================================ consumer warps
  const int lane = tid & 31;
  int st = 0;
  uint32_t par = 0;
  const unsigned char* base = smem;  // the next stage

  for (long long item = blockIdx.x; item < b.nitems; item += gridDim.x) {
    const int gi = find_group(b, item);
    const GroupDev& G = b.g[gi];
    int sl = 0, tile = (int)(item - G.item0);
    if (!GRAD) item_coords32(b, G, item - G.item0, sl, tile);
    SysDev* sd = (MODE == M_APPLY) ? nullptr : b.sys + (G.sys0 + sl);
    if (MODE != M_APPLY && skip_item(sd)) continue;

    const int nx = G.nx, ny = G.ny, nz = G.nz, npml = G.npml;
    const int plane = nx * ny;
    const int z0 = (tile % G.zsplit) * G.zc, z1 = min(z0 + G.zc, nz);
    const int c0 = (tile / G.zsplit) * G.chunk, c1 = min(c0 + G.chunk, plane);
    const bool edge = c0 < nx || c1 + nx > plane;  // some y neighbour lies outside the plane
    long long off = (long long)sl * G.n;
    const int iter = HASB ? sd->iter : 0;
    const R om2 = pick<R>(G.om2, G.om2f);
    const R ih2 = pick<R>(G.ih2, G.ih2f);
    const R* tab = (MODE == M_APPLY) ? s_tab : (sizeof(R) == 4 ? (const R*)G.ltab32 : (const R*)G.ltab64);

    // this thread's nodes
    const int e0 = c0 + (PAIR ? 2 * tid : tid);
    bool own[NPT];
    int ni[NPT], nj[NPT];
    uint32_t rcb = 0;      // the thread's columns that hold receivers of this system
    uint32_t rz[NPT] = {};  // their receivers at the current 32 planes
    bool gen = false;   // a stretched axis or a neighbour outside the grid
    bool geny = false;  // the y axis too
#pragma unroll
    for (int r = 0; r < NPT; ++r) {
      own[r] = e0 + r * RS < c1;
      const int ee = own[r] ? e0 + r * RS : c0;
      nj[r] = ee / nx;
      ni[r] = ee - nj[r] * nx;
      const int w = npml > 0 ? npml + 1 : 1;
      geny = geny || (own[r] && !(nj[r] >= w && nj[r] < ny - w));
      gen = gen || geny || (own[r] && !(ni[r] >= w && ni[r] < nx - w));
      if (NORM && G.rmask && own[r]) {
        if ((__ldg(G.rcol + ((long long)sl * ny + nj[r]) * G.rw + (ni[r] >> 5)) >> (ni[r] & 31)) & 1u) rcb |= 1u << r;
      }
    }
    gen = __any_sync(0xffffffffu, gen);
    if (XO) geny = __any_sync(0xffffffffu, geny);
    const bool idle = !__any_sync(0xffffffffu, own[0]);  // the warp lies past the chunk's end

    const R coef = MODE == M_P1 ? (iter > 0 ? R(sd->beta) : R(0)) : MODE == M_P2 ? -R(sd->alpha) : R(0);
    int src_k = -1, src_r = -1;  // plane of the source, and which of the thread's nodes it is
    C a_src = czero<R>();
    auto load_src = [&]() {
      src_k = (int)(sd->src / plane);
      const int d = (int)(sd->src - (long long)src_k * plane) - e0;
      src_r = d == 0 ? 0 : (NPT > 1 && d == RS) ? 1 : -1;
      if ((MODE == M_RES || GRAD) && G.alpha) a_src = mkc(R(G.alpha[2 * sl]), R(G.alpha[2 * sl + 1]));
    };
    if ((MODE == M_P1 && G.masked) || MODE == M_RES || GRAD) load_src();

    // running addresses: F is stored at plane k, the output at plane k - 1
    C* pF = nullptr;
    if (MODE == M_P1) pF = (C*)G.p[pslot(b, iter)] + off + (long long)z0 * plane + e0;
    if (MODE == M_P2) pF = (C*)G.r1[(iter & 1) ^ 1] + off + (long long)z0 * plane + e0;
    // (the first step's "plane z0 - 1" is nobody's: it goes to plane z0, which the next step writes)
    OC* pO = (OC*)(MODE == M_P1 ? G.t1 : MODE == M_RES ? G.r1[0] : G.s) + off + (long long)z0 * plane + e0;
    // bytes from the region's start to its first node (c0 - nx) and to the model's (c0): the copies start at
    // 16-byte boundaries, so these change with the plane when its bytes are not a multiple of 16
    constexpr bool SHIFT = !PAIR && CB == 8;
    const int em = G.m_double ? 8 : 4;
    const long long pofs = ((long long)(z0 - 1) * plane + c0 - nx) * CB;
    uint32_t da = SHIFT ? (uint32_t)(((uintptr_t)field_a(G, iter) + (long long)sl * G.n * CB + pofs) & 15) : 0u;
    uint32_t db = SHIFT && HASB ? (uint32_t)(((uintptr_t)field_b(G, iter) + (long long)sl * G.n * CB + pofs) & 15) : 0u;
    uint32_t dm = (uint32_t)(((uintptr_t)G.m + ((long long)z0 * plane + c0) * em) & 15);
    const uint32_t pstep = (uint32_t)(((long long)plane * CB) & 15), mstep = (uint32_t)(((long long)plane * em) & 15);
    const int o = nx + (PAIR ? 2 * tid : tid);  // own (first) node in the region

    // coefficients of the thread's nodes (only warps with a stretched or boundary node)
    constexpr int NY = PAIR ? 1 : NPT;  // rows of the thread's nodes (a pair lies in one row)
    C am[NPT], ap[NPT], bm[NY], bp[NY];
    R sx_[NPT], sy_[NY];
    R w2xy[NPT];  // gradient: |s_x s_y|^2

    double accd = 0.0;
    // sum of |output|^2: FP32 over 4 planes, then FP64 (pairs past the chunk's end are left out at the end)
    R accf = R(0);
    C fc[NPT], q[NPT];
    C zm[NPT];  // complex128: the z - 1 neighbour of a pending plane off the z layers
#pragma unroll
    for (int r = 0; r < NPT; ++r) fc[r] = q[r] = zm[r] = czero<R>();
    C hz = mkc(ih2, R(0));  // weight of the z + 1 neighbour of the pending plane
    R hs = R(0);            // gradient: Im s_z of the pending plane
    if constexpr (GRAD)
      for (int k = 0; k < z1 - z0; ++k)
#pragma unroll
        for (int r = 0; r < NPT; ++r) gacc[k * L + tid + r * NC] = 0.0;

    auto wait = [&]() -> bool {
      if (mbar_try_wait(&full[st], par)) return true;
      if (mbar_wait_or_abort(&full[st], par, &s_abort, T.wait_ns)) return true;
      s_abort = 1;
      if (T.err) atomicExch(T.err, 1);
      return false;
    };
    auto release = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
      base += SB;
      if (++st == S) {
        st = 0;
        base = smem;
        par ^= 1;
      }
      if (SHIFT) {
        da = (da + pstep) & 15;
        db = (db + pstep) & 15;
      }
    };
    // F of this thread's nodes in the current stage
    auto own_f = [&](const C* A, const C* B, C (&v)[NPT]) {
      if constexpr (PAIR) {
        const float4 a = ld4(A);
        v[0] = lo2(a);
        v[1] = hi2(a);
        if (HASB) {
          const float4 bb = ld4(B);
          v[0] = rfma(coef, lo2(bb), v[0]);
          v[1] = rfma(coef, hi2(bb), v[1]);
        }
      } else {
#pragma unroll
        for (int r = 0; r < NPT; ++r) {
          v[r] = A[r * RS];
          if (HASB) v[r] = rfma(coef, B[r * RS], v[r]);
        }
      }
    };
    // gradient: the finished plane kp, accumulated over the systems.  t is the stencil without the node factor
    // w = s_x s_y s_z, which leaves the sums: with A u - c = w t', t' = t - c / w,
    //   Re(conj(w u) w t') = |w|^2 Re(conj(u) t'),  |w t'|^2 = |w|^2 |t'|^2,
    // and |w|^2 enters the gradient once, after the last system: 9 to 12 FP64 instructions less per node and
    // system in the layer, 22 % of the time on 148^3 x 16.
    auto accum = [&](int kp, C (&t)[NPT], bool g, bool z) {
#pragma unroll
      for (int r = 0; r < NPT; ++r) {
        if (!own[r]) continue;
        if (G.q || (kp == src_k && r == src_r)) {
          const C c = G.q ? q_at<R>(G, sl, (long long)kp * plane + e0 + r * RS) : a_src;
          C w = mkc(R(1), g ? sx_[r] : R(0));
          if (g) w = smul(sy_[r], w);
          if (z) w = smul(hs, w);
          const R d = R(1) / abs2(w);
          t[r] = t[r] - mkc((c.x * w.x + c.y * w.y) * d, (c.y * w.x - c.x * w.y) * d);
        }
        double* ga = gacc + (kp - z0) * L + tid + r * NC;
        *ga = fma_r(fc[r].x, t[r].x, fma_r(fc[r].y, t[r].y, *ga));
        if (g || z) {
          const R w2 = (g ? w2xy[r] : R(1)) * (z ? fma_r(hs, hs, R(1)) : R(1));
          accd = fma_r(w2, fma_r(t[r].x, t[r].x, t[r].y * t[r].y), accd);
        } else {
          accd = fma_r(t[r].x, t[r].x, fma_r(t[r].y, t[r].y, accd));
        }
      }
    };
    // the finished stencil t of plane kp: mask, right-hand side, store, norm
    auto emit = [&](int kp, C (&t)[NPT]) {
      if (MODE == M_P1 && kp == src_k) {
#pragma unroll
        for (int r = 0; r < NPT; ++r)
          if (r == src_r) t[r] = czero<R>();
      }
      if (MODE == M_RES) {
#pragma unroll
        for (int r = 0; r < NPT; ++r) {
          C rr = mkc(-t[r].x, -t[r].y);
          if (G.q) {
            if (own[r] && kp >= z0) rr = q_at<R>(G, sl, (long long)kp * plane + e0 + r * RS) - t[r];
          } else if (kp == src_k && r == src_r) {
            rr = G.masked ? czero<R>() : a_src - t[r];
          }
          t[r] = rr;
        }
      }
      if (GV) {
        // refinement inner solve: s = S^H r + S^H r64
        const float2* pG = (const float2*)G.gvec + (pO - (OC*)G.s);
        if constexpr (PAIR) {
          if (own[0]) {
            const float4 gv = __ldg(reinterpret_cast<const float4*>(pG));
            t[0] = t[0] + lo2(gv);
            t[1] = t[1] + hi2(gv);
          }
        } else {
#pragma unroll
          for (int r = 0; r < NPT; ++r)
            if (own[r]) t[r] = t[r] + to_c(__ldg(pG + r * RS), R(0));
        }
      }
      uint32_t skip = 0;
      if ((MODE == M_P2 || MODE == M_SH) && rcb) {
        // receivers of this plane: left to the finalizer (rec_col_bits), or (FP64 normal residual of the
        // refinement, where A^H F and lambda P^T r2 nearly cancel) added here before the one rounding
        if (kp == z0 || (kp > z0 && (kp & 31) == 0)) {
#pragma unroll
          for (int r = 0; r < NPT; ++r)
            rz[r] = ((rcb >> r) & 1u) ? __ldg(G.rmask + ((long long)sl * plane + e0 + r * RS) * G.zw + (kp >> 5)) : 0u;
        }
#pragma unroll
        for (int r = 0; r < NPT; ++r)
          if (kp >= z0 && ((rz[r] >> (kp & 31)) & 1u)) {
            if (MODE == M_SH && G.rmap) {
              const int rk = G.rmap[off + (long long)kp * plane + e0 + r * RS];
              t[r] = t[r] + R(G.lambda) * ((const C*)b.r2)[rk];
            } else {
              skip |= 1u << r;
            }
          }
      }
      if constexpr (PAIR && sizeof(OR) == 4) {
        if (own[0]) st4(pO, t[0], t[1]);
      } else {
#pragma unroll
        for (int r = 0; r < NPT; ++r)
          if (own[r]) {
            if constexpr (sizeof(R) == 8 && sizeof(OR) == 4) pO[r * RS] = mkc(narrow(t[r].x), narrow(t[r].y));
            else pO[r * RS] = to_c(t[r], OR(0));
          }
      }
      pO += plane;
      // FP64: straight into the sum (three additions of zero less).  With the model and the complex64 output
      // converted in integers this took 11 % off M_SH and 4 % off M_RES (116^3 x 32).
      if (NORM && sizeof(R) == 8) {
#pragma unroll
        for (int r = 0; r < NPT; ++r)
          if (own[r] && !((skip >> r) & 1u)) accd = fma_r(t[r].x, t[r].x, fma_r(t[r].y, t[r].y, accd));
      } else if (NORM) {
        R s2 = R(0);
#pragma unroll
        for (int r = 0; r < NPT; ++r) {
          const R a2 = fma_r(t[r].x, t[r].x, t[r].y * t[r].y);
          s2 += (((skip >> r) & 1u) || !(PAIR || own[r])) ? R(0) : a2;
        }
        accf += s2;
        if ((kp & 3) == 3) {
          accd += (double)accf;
          accf = R(0);
        }
      }
    };
    if (gen) {
#pragma unroll
      for (int r = 0; r < NPT; ++r) {
        const AxisCoef<R> cx_ = axis_coef<R, CONJ>(tab, ni[r], nx, npml, ih2);
        const AxisCoef<R> cy_ = axis_coef<R, CONJ>(tab, nj[r], ny, npml, ih2);
        am[r] = cx_.am;
        ap[r] = cx_.ap;
        if (r < NY) {
          bm[r] = cy_.am;
          bp[r] = cy_.ap;
          sy_[r] = cy_.im;
        }
        w2xy[r] = fma_r(cx_.im, cx_.im, R(1)) * fma_r(cy_.im, cy_.im, R(1));
        sx_[r] = cx_.im;
      }
    }
    // One plane of the item: its F, the z + 1 term of plane k - 1, and its own stencil without that term.
    // gen_c: 1 the x coefficients are general, 2 those of x and y; zg_c: plane k lies in a z layer.  XO (FP64)
    // has a kind of its own for x alone, with 8 FP64 instructions of 37 less (the phases 6: their kernels with
    // and without it round alike): of the warps of 81^3 two thirds have an x layer, of 148^3 a third, most of
    // them outside the y layers.  The phases take it for items of 8 planes and more, where the additional loops
    // pay: us per iteration without and with it, items of 2 and 3 planes 39.3 / 40.7 (36^3 x 1) and 127.0 / 125.2
    // (48^3 x 4), of 9 to 50 planes 923 / 878 (81^3 x 9), 493 / 479 (84^3 x 4), 1181 / 1141 (116^3 x 4), 609 / 589
    // (148^3 x 1) and 141.4 / 142.4 (81^3 x 1).  Nothing between 3 and 9 planes was measured.
    auto step = [&](auto gen_c, auto zg_c, int k) -> bool {
      constexpr bool GEN = decltype(gen_c)::value > 0, GY = decltype(gen_c)::value == 2, ZG = decltype(zg_c)::value;
      if (!wait()) return false;
      const C* A = reinterpret_cast<const C*>(base + da) + o;
      const C* B = HASB ? reinterpret_cast<const C*>(base + db + T.off_b) + o : nullptr;
      C v[NPT];
      own_f(A, B, v);
      if (HASB) {
        if constexpr (PAIR) {
          if (own[0]) st4(pF, v[0], v[1]);
        } else {
#pragma unroll
          for (int r = 0; r < NPT; ++r)
            if (own[r]) pF[r * RS] = v[r];
        }
        pF += plane;
      }
      // in-plane neighbours
      C l[NPT], rgt[NPT], ym[NPT], yp[NPT];
      R mk[NPT];
      const unsigned char* Mp = base + (T.off_m + dm);
      dm = (dm + mstep) & 15;
      if constexpr (PAIR) {
        const float2 m2 = *reinterpret_cast<const float2*>(Mp + 8 * tid);
        mk[0] = m2.x;
        mk[1] = m2.y;
        C ll = A[-1], rr = A[2];
        const float4 am4 = ld4(A - nx), ap4 = ld4(A + nx);
        ym[0] = lo2(am4);
        ym[1] = hi2(am4);
        yp[0] = lo2(ap4);
        yp[1] = hi2(ap4);
        if (HASB) {
          ll = rfma(coef, B[-1], ll);
          rr = rfma(coef, B[2], rr);
          const float4 bm4 = ld4(B - nx), bp4 = ld4(B + nx);
          ym[0] = rfma(coef, lo2(bm4), ym[0]);
          ym[1] = rfma(coef, hi2(bm4), ym[1]);
          yp[0] = rfma(coef, lo2(bp4), yp[0]);
          yp[1] = rfma(coef, hi2(bp4), yp[1]);
        }
        l[0] = ll;
        rgt[0] = v[1];
        l[1] = v[0];
        rgt[1] = rr;
      } else {
#pragma unroll
        for (int r = 0; r < NPT; ++r) {
          const int x = r * RS;
          mk[r] = model_smem<R>(Mp, G.m_double, tid + x);
          l[r] = A[x - 1];
          rgt[r] = A[x + 1];
          ym[r] = A[x - nx];
          yp[r] = A[x + nx];
          if (HASB) {
            l[r] = rfma(coef, B[x - 1], l[r]);
            rgt[r] = rfma(coef, B[x + 1], rgt[r]);
            ym[r] = rfma(coef, B[x - nx], ym[r]);
            yp[r] = rfma(coef, B[x + nx], yp[r]);
          }
        }
      }
      if (DUMMY || k > z0) {
        C t[NPT];
#pragma unroll
        for (int r = 0; r < NPT; ++r) {
          if (ZG) t[r] = cfma(hz, v[r] - fc[r], q[r]);
          else t[r] = rfma(ih2, DIFF ? v[r] - fc[r] : rfma(R(-2), fc[r], zm[r] + v[r]), q[r]);
          if (GEN && !GRAD) t[r] = smul(sx_[r], t[r]);
          if (GY && !GRAD) t[r] = smul(sy_[PAIR ? 0 : r], t[r]);
        }
        if constexpr (GRAD) {
          accum(k - 1, t, GEN, ZG);
        } else {
          emit(k - 1, t);
        }
      }
      AxisCoef<R> cz;
      if (ZG) {
        cz = axis_coef<R, CONJ>(tab, k, nz, npml, ih2, &hz);
        if (GRAD) {
          hz = cz.ap;
          hs = cz.im;
        }
      }
#pragma unroll
      for (int r = 0; r < NPT; ++r) {
        if (GEN) {
          // outside the grid: zero (the stage holds other rows or nothing there)
          // (of a pair in a row of even length only the first node can lie at its start, the second at its end)
          if (!(PAIR && r == 1) && ni[r] == 0) l[r] = czero<R>();
          if (!(PAIR && r == 0) && ni[r] == nx - 1) rgt[r] = czero<R>();
          if (edge) {
            if (nj[PAIR ? 0 : r] == 0) ym[r] = czero<R>();
            if (nj[PAIR ? 0 : r] == ny - 1) yp[r] = czero<R>();
          }
        }
        if (DIFF) {
          l[r] = l[r] - v[r];
          rgt[r] = rgt[r] - v[r];
          ym[r] = ym[r] - v[r];
          yp[r] = yp[r] - v[r];
        }
        const R c = om2 * mk[r];
        C acc;
        if (DIFF) {
          const C dz = fc[r] - v[r];
          acc = mkc(c * v[r].x, c * v[r].y);
          if (GEN) {
            acc = cfma(am[r], l[r], acc);
            acc = cfma(ap[r], rgt[r], acc);
            acc = GY ? cfma(bm[PAIR ? 0 : r], ym[r], acc) : rfma(ih2, ym[r], acc);
            acc = GY ? cfma(bp[PAIR ? 0 : r], yp[r], acc) : rfma(ih2, yp[r], acc);
            acc = ZG ? cfma(cz.am, dz, acc) : rfma(ih2, dz, acc);
          } else {
            C sum = (l[r] + rgt[r]) + (ym[r] + yp[r]);
            if (!ZG) sum = sum + dz;
            acc = rfma(ih2, sum, acc);
            if (ZG) acc = cfma(cz.am, dz, acc);
          }
        } else {
          // In a z layer every term but omega^2 m u is a difference: these first, then that one in one rounding.
          // The phases have kernels with and without the loops for x alone (XO), which have to round alike.
          constexpr bool YD = GY || (GEN && HASB);
          acc = ZG ? cmul(cz.am, fc[r] - v[r]) : mkc(c * v[r].x, c * v[r].y);
          if (!GEN && !ZG) {
            acc = rfma(ih2, rfma(R(-4), v[r], (l[r] + rgt[r]) + (ym[r] + yp[r])), acc);
          } else {
            if (GEN) acc = cfma(ap[r], rgt[r] - v[r], cfma(am[r], l[r] - v[r], acc));
            else acc = rfma(ih2, rfma(R(-2), v[r], l[r] + rgt[r]), acc);
            if (GY) acc = cfma(bp[r], yp[r] - v[r], cfma(bm[r], ym[r] - v[r], acc));
            else if (YD) acc = rfma(ih2, yp[r] - v[r], rfma(ih2, ym[r] - v[r], acc));
            else acc = rfma(ih2, rfma(R(-2), v[r], ym[r] + yp[r]), acc);
          }
          if (ZG) acc = rfma(c, v[r], acc);
          zm[r] = fc[r];
        }
        q[r] = ZG && !GRAD ? smul(cz.im, acc) : acc;
        fc[r] = v[r];
      }
      if (DUMMY && k == z0) {  // what this step finished was no plane of the item
        pO -= plane;
        accf = R(0);
        accd = 0.0;
      }
      release();
      return true;
    };
    // the planes of the item: low z layer, interior, high z layer
    auto planes = [&](auto gen_c) -> bool {
      const int za = npml > 0 ? min(z1, npml + 1) : z0, zb = npml > 0 ? min(z1, nz - 1 - npml) : z1;
      int k = z0;
      for (; k < za; ++k)
        if (!step(gen_c, std::true_type(), k)) return false;
      const int kl = k;
      // complex128: a pending plane of the layer (where 1 / s(half) = 1) lacks (up - u) / h^2 alone
      if (!DIFF && k < zb) {
#pragma unroll
        for (int r = 0; r < NPT; ++r) zm[r] = fc[r];
      }
      for (; k < zb; ++k)
        if (!step(gen_c, std::false_type(), k)) return false;
      if (k > kl) {  // the pending plane is an interior one
        hz = mkc(ih2, R(0));
        hs = R(0);
        if (!DIFF) {
#pragma unroll
          for (int r = 0; r < NPT; ++r) q[r] = rfma(ih2, zm[r] - fc[r], q[r]);
        }
      }
      for (; k < z1; ++k)
        if (!step(gen_c, std::true_type(), k)) return false;
      return true;
    };

    bool dead = false;
    const int passes = GRAD ? G.nsys : 1;
    for (int pass = 0; pass < passes && !dead; ++pass) {
      if (GRAD && pass > 0) {  // the next system of the group
        ++sl;
        ++sd;
        off += G.n;
        load_src();
        da = SHIFT ? (uint32_t)(((uintptr_t)field_a(G, 0) + (long long)sl * G.n * CB + pofs) & 15) : 0u;
        dm = (uint32_t)(((uintptr_t)G.m + ((long long)z0 * plane + c0) * em) & 15);
        hz = mkc(ih2, R(0));
        hs = R(0);
#pragma unroll
        for (int r = 0; r < NPT; ++r) fc[r] = q[r] = czero<R>();
      }
      if (z0 > 0) {  // the plane below gives the z - 1 neighbours
        if (wait()) {
          own_f(reinterpret_cast<const C*>(base + da) + o,
                HASB ? reinterpret_cast<const C*>(base + db + T.off_b) + o : nullptr, fc);
          release();
        } else {
          dead = true;
        }
      } else if (SHIFT) {
        da = (da + pstep) & 15;
        db = (db + pstep) & 15;
      }
      if (idle) {
        for (int k = z0; k < z1 && !dead; ++k) {
          dead = !wait();
          if (!dead) release();
        }
      } else if (!dead) {
        if (!gen) {
          dead = !planes(std::integral_constant<int, 0>());
        } else if (XO && !geny) {
          if constexpr (XO) dead = !planes(std::integral_constant<int, 1>());
        } else {
          dead = !planes(std::integral_constant<int, 2>());
        }
      }
      if (!dead) {
        // the plane above completes the last one
        C v[NPT];
#pragma unroll
        for (int r = 0; r < NPT; ++r) v[r] = czero<R>();
        if (z1 < nz) {
          if (wait()) {
            own_f(reinterpret_cast<const C*>(base + da) + o,
                  HASB ? reinterpret_cast<const C*>(base + db + T.off_b) + o : nullptr, v);
            release();
          } else {
            dead = true;
          }
        }
        if (!dead) {
          C t[NPT];
#pragma unroll
          for (int r = 0; r < NPT; ++r) {
            t[r] = cfma(hz, v[r] - fc[r], q[r]);
            if (gen && !GRAD) t[r] = smul(sy_[PAIR ? 0 : r], smul(sx_[r], t[r]));
          }
          if constexpr (GRAD) accum(z1 - 1, t, gen, true);
          else emit(z1 - 1, t);
        }
      }
    }
    if (sizeof(R) == 4) accd = PAIR && !own[0] ? 0.0 : accd + (double)accf;


    if (MODE == M_APPLY) {
      if (!dead) continue;
      // no error flag to raise: the time-out (which a complete set of copies cannot reach) shows as NaN
#pragma unroll
      for (int r = 0; r < NPT; ++r)
        if (own[r])
          for (int k = z0; k < z1; ++k) ((OC*)G.s)[off + (long long)k * plane + e0 + r * RS] = mkc(OR(NAN), OR(NAN));
      break;
    }
    // ---- item partial, ticket and the system's finalizer (consumer threads only)
    const double tsum = block_sum<NC, CSync>(accd, red);
    if (GRAD) {
      if (first_threads_any<NC>(dead || s_abort != 0)) {
        // no error flag to raise: the time-out (which a complete set of copies cannot reach) shows as NaN
        if (tid == 0) atomicAdd(b.f, (double)NAN);
        break;
      }
      for (int k = z0; k < z1; ++k) {
        const R im = axis_coef<R, false>(tab, k, nz, npml, ih2).im;
        const R w2z = om2 * fma_r(im, im, R(1));
#pragma unroll
        for (int r = 0; r < NPT; ++r)
          if (own[r])
            G.grad[(long long)k * plane + e0 + r * RS] += (gen ? w2xy[r] : R(1)) * w2z * gacc[(k - z0) * L + tid + r * NC];
      }
      if (tid == 0 && tsum != 0.0) atomicAdd(b.f, 0.5 * tsum);
      continue;
    }
    // the copy warp may raise the flag at any time: decide on one reduced value
    if (first_threads_any<NC>(s_abort != 0)) break;
    if (tid == 0 && NORM) b.partial[sd->part_off + tile] = tsum;
    // what the finalizing CTA reads of this one: the partial sum, and p or s at the receivers
    if (tid == 0 || rcb) __threadfence();
    CSync::sync();
    if (tid == 0) {
      const unsigned t = atomicAdd(&sd->ticket, 1u);
      s_last = (t == (unsigned)(G.ntiles - 1));
      __threadfence();
    }
    CSync::sync();
    if (s_last) finalize_lin<R, OR, MODE, NC, CSync>(b, G, sd, sl, red);
  }
}

// ------------------------------------------------------------------ start of a solve
// (A^H)[node, src] of the point field e_src: the stencil weight of src in the row of a node that is src or
// one of its six neighbours.
template <typename R>
__device__ cx<R> point_weight(const GroupDev& G, const R* tab, long long node, int di, int dj, int dk) {
  typedef cx<R> C;
  const long long plane = (long long)G.nx * G.ny;
  const int k = (int)(node / plane);
  const int rem = (int)(node - (long long)k * plane);
  const int j = rem / G.nx, i = rem - j * G.nx;
  const R ih2 = inv_h2<R>(G);
  const AxisCoef<R> cx_ = axis_coef<R, true>(tab, i, G.nx, G.npml, ih2);
  const AxisCoef<R> cy_ = axis_coef<R, true>(tab, j, G.ny, G.npml, ih2);
  const AxisCoef<R> cz_ = axis_coef<R, true>(tab, k, G.nz, G.npml, ih2);
  C w;
  if (di) w = di < 0 ? cx_.am : cx_.ap;
  else if (dj) w = dj < 0 ? cy_.am : cy_.ap;
  else if (dk) w = dk < 0 ? cz_.am : cz_.ap;
  else {
    w = cx_.a0 + cy_.a0 + cz_.a0;
    w.x += pick<R>(G.omega * G.omega, G.om2f) * model_at<R>(G.m, G.m_double, node);
  }
  return smul(cx_.im, smul(cy_.im, smul(cz_.im, w)));
}

// s = S^H b for a point right-hand side b1 = alpha e (or 0) and b2 = lambda d, without a pass over the
// grid: A^H b1 is non-zero at the source and its neighbours only.  One block of 128 threads per system;
// the caller zeroed s and r1 (cold start; the reference norm of a warm start, SH_REF, needs no zeroed
// vector).  Flavors and scalars as the stencil pass M_SH.
template <typename R, typename OR>
__global__ void k_init_point(const __grid_constant__ Batch b, int nsys_total) {
  typedef cx<R> C;
  typedef cx<OR> OC;
  __shared__ double red[4];
  __shared__ long long pn[7];
  __shared__ C pv[7];
  __shared__ int prec[7];  // the node is a receiver too
  const int s = blockIdx.x;
  if (s >= nsys_total) return;
  SysDev* sd = b.sys + s;
  const GroupDev& G = b.g[sd->group];
  const long long off = (long long)sd->local * G.n;
  const int t = threadIdx.x;
  C a = czero<R>();
  if (G.alpha) a = mkc(R(G.alpha[2 * sd->local]), R(G.alpha[2 * sd->local + 1]));
  if (t < 7) {
    // node t of the source's stencil, and the direction from it to the source
    const int di = t == 1 ? 1 : t == 2 ? -1 : 0, dj = t == 3 ? 1 : t == 4 ? -1 : 0, dk = t == 5 ? 1 : t == 6 ? -1 : 0;
    const long long plane = (long long)G.nx * G.ny;
    const int k = (int)(sd->src / plane) - dk;
    const int rem = (int)(sd->src % plane);
    const int j = rem / G.nx - dj, i = rem % G.nx - di;
    const bool in = G.alpha && i >= 0 && i < G.nx && j >= 0 && j < G.ny && k >= 0 && k < G.nz;
    pn[t] = in ? (long long)k * plane + (long long)j * G.nx + i : -1;
    pv[t] = czero<R>();
    prec[t] = 0;
    if (in) {
      pv[t] = point_weight<R>(G, sizeof(R) == 4 ? (const R*)G.ltab32 : (const R*)G.ltab64, pn[t], di, dj, dk) * a;
      ((OC*)G.s)[off + pn[t]] = to_c(pv[t], OR(0));
    }
    if (t == 0 && G.alpha && b.flavor == SH_INIT) ((C*)G.r1[0])[off + sd->src] = a;
  }
  __syncthreads();
  // ||s||^2: the source's nodes, then the receivers (a receiver among the former counts once, with both terms)
  double acc = 0.0;
  const C* r2 = (const C*)b.r2;
  for (int k = sd->rec_begin + t; k < sd->rec_end; k += blockDim.x) {
    const long long node = b.rec_idx[k];
    C v = R(G.lambda) * r2[k];
    for (int p = 0; p < 7; ++p)
      if (pn[p] == node) {
        v = v + pv[p];
        prec[p] = 1;
      }
    const OC sv = to_c(v, OR(0));
    ((OC*)G.s)[off + node] = sv;
    acc += G.rmap ? (double)abs2(v) : (double)abs2(sv);
  }
  __syncthreads();
  if (t < 7 && pn[t] >= 0 && !prec[t]) acc += (double)abs2(pv[t]);
  acc = block_sum<128>(acc, red);
  if (t == 0) {
    sh_scalars(b, sd, acc);
    sd->ticket = 0u;
  }
}

// r1[src] = alpha for every system of a group (r1 zeroed before).
template <typename R>
__global__ void k_point_field(const __grid_constant__ Batch b, int gi) {
  const GroupDev& G = b.g[gi];
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < G.nsys)
    ((cx<R>*)G.r1[0])[(long long)s * G.n + b.sys[G.sys0 + s].src] = mkc(R(G.alpha[2 * s]), R(G.alpha[2 * s + 1]));
}

// ------------------------------------------------------------------ iterate updates
// x += alpha_{k-m} p_{k-m} + ... + alpha_{k-1} p_{k-1}, after every m-th iteration (m = b.xsteps; the
// directions wait in the ring of slots, which the next phase 1 starts to overwrite), and the steps left
// over of a system that has stopped.  The oldest step is added first, so x rounds as with one update per
// iteration.  A pass of its own: 16 + 8 m bytes per node and m iterations at the speed of a copy (the
// phases keep their registers and their shared memory for planes).  NV nodes per access.
template <typename R, int NV>
__global__ void __launch_bounds__(256) k_xupdate(const __grid_constant__ Batch b) {
  struct alignas(sizeof(R) * 2 * NV) V {
    R v[2 * NV];
  };
  const int m = b.xsteps;
  for (long long item = blockIdx.x; item < b.xitems; item += gridDim.x) {
    int gi = 0;
    while (gi < b.ngroups - 1 && item >= b.g[gi + 1].xitem0) ++gi;
    const GroupDev& G = b.g[gi];
    const int per = (int)((G.n + kXupdNodes - 1) / kXupdNodes);
    const int sl = (int)((item - G.xitem0) / per), part = (int)((item - G.xitem0) % per);
    SysDev* sd = b.sys + (G.sys0 + sl);
    const int state = sd->state, iter = sd->iter;
    if (state == ST_DONE || (state == ST_ACTIVE && (iter == 0 || iter % m != 0))) continue;
    const int c = iter > 0 ? (iter - 1) % m + 1 : 0;  // steps not yet in x: iterations iter - c .. iter - 1
    const long long n0 = (long long)part * kXupdNodes, n1 = min(n0 + kXupdNodes, G.n);
    V* X = (V*)((cx<R>*)G.x + (long long)sl * G.n);
    const V* P[4];
    R h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      // i counts back from the newest step
      P[i] = (const V*)((const cx<R>*)G.p[pslot(b, iter - 1 - i)] + (long long)sl * G.n);
      h[i] = i < c ? R(i == 0 ? sd->alpha : sd->alpha_hist[i - 1]) : R(0);
    }
    for (long long v = n0 / NV + threadIdx.x; v < n1 / NV; v += 256) {
      V x = X[v], p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < c) p[i] = P[i][v];
#pragma unroll
      for (int i = 3; i >= 0; --i)
        if (i < c) {
#pragma unroll
          for (int w = 0; w < 2 * NV; ++w) x.v[w] = fma_r(h[i], p[i].v[w], x.v[w]);
        }
      X[v] = x;
    }
    if (state == ST_FINISHING) {
      // the last part of the system closes it
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&sd->ticket, 1u) == (unsigned)(per - 1)) {
          sd->ticket = 0u;
          sd->state = ST_DONE;
          atomicSub(b.remaining, 1);
        }
      }
    }
  }
}

}  // namespace wri
