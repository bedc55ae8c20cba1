// amrfd_kernels.cu -- FP64 kernels of the FD-MP5 update (Porth et al. 2014, Sec. 2).
//
//  speeds_kernel   maximal characteristic speed per cell -> per-domain c_max per
//                  direction (Sec. 2.2, "grid-global c_max") and the CFL rate
//                  sum_d c_d/dx_d (Sec. 4.4); exact IEEE operations in the order
//                  of the definition, reduced with integer max on the bit patterns.
//  flux_kernel     one direction's flux difference for a tile of lines:
//                  halo synthesis (periodic / zero-gradient / mirror), the stored
//                  derived quantities, physical flux, Lax-Friedrichs split
//                  G^{+-} = F +- c_max U (Sec. 2.2) into shared memory, then MP5 (or
//                  LIMO3) at every face (Suresh & Huynh 1997, as cited in Sec. 2.2) on
//                  both biases, F^ = R_L(F^+) + R_R(F^-), and -dF^/dx (Sec. 2.1); the
//                  sweeps run in parts, the costliest variable's on a spare warp.
//  combine_kernel  Shu-Osher stage U^(i) = sum a U^(k) + dt b L (Sec. 2.3), GLM psi
//                  damping after the last stage (Sec. 4.2), speeds of U^(i).
//  dt_kernel       dt = CFL / rate per domain, clamped to t_end - t.
//  compact kernels device-side work list of the active blocks (App. C).
#include <cuda_runtime.h>

#include "amrfd_device.cuh"
#include "amrfd_kernels.cuh"
#include "amrfd_sweep.cuh"

namespace amrfd {

// ----------------------------------------------------------------- utilities
__device__ __forceinline__ void block_coords(const DomDev& dm, int blk, int o[3]) {
  int bx = blk % dm.nb[0];
  int by = (blk / dm.nb[0]) % dm.nb[1];
  int bz = blk / (dm.nb[0] * dm.nb[1]);
  o[0] = bx * dm.be[0];
  o[1] = by * dm.be[1];
  o[2] = bz * dm.be[2];
}

__device__ __forceinline__ DomDev load_dom(const DomDev* p) { return *p; }

// block-wide max of four u64 values; result valid in thread 0
__device__ __forceinline__ void block_max4(unsigned long long v[4], unsigned long long (*red)[32]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    unsigned long long x = warp_max_u64(v[q]);
    if (lane == 0) red[q][wid] = x;
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      unsigned long long x = lane < nw ? red[q][lane] : 0ull;
      v[q] = warp_max_u64(x);
    }
  }
  __syncthreads();
}

// block-wide max of four non-negative floats, broadcast to every thread
__device__ __forceinline__ void block_max4f_bcast(float v[4], float (*redf)[32], float* out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    float x = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    if (lane == 0) redf[q][wid] = x;
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      float x = lane < nw ? redf[q][lane] : 0.0f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
      if (lane == 0) out[q] = x;
    }
  }
  __syncthreads();
}

// Exact speeds of one cell folded into the running maxima (IEEE operations in the
// order of the definition); returns false for a non-physical state.
template <int PHYS, int NV>
__device__ __forceinline__ bool exact_speeds(const double* u, double gamma, int ndim, const double* dx, bool want_rate,
                                             unsigned long long mx[4]) {
  Prim w;
  if (!cons2prim_exact<PHYS, NV>(u, gamma, ndim, w)) return false;
  double rate = 0.0;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    if (d < ndim) {
      const double cd = char_speed_exact<PHYS>(w, gamma, d);
      const unsigned long long b = (unsigned long long)dbits(cd);
      mx[d] = b > mx[d] ? b : mx[d];
      if (want_rate) rate = __dadd_rn(rate, __ddiv_rn(cd, dx[d]));
    }
  }
  const unsigned long long br = (unsigned long long)dbits(rate);
  mx[3] = br > mx[3] ? br : mx[3];
  return true;
}

// ------------------------------------------------------------------ speeds
// Exact per-domain maxima in two launches. The bounds launch (exact = 0) evaluates
// FP32 bounds of every active cell's speeds and publishes, per domain, the largest
// lower bound T (an integer max of the FP32 bits), and per item the largest upper bound
// (+inf when a cell carries none). The exact launch (exact = 1) skips the items whose
// upper bounds stay below T, re-evaluates the bounds of the other items' cells and
// computes the exact IEEE speeds only of the cells whose upper bound reaches T, or that
// carry no bound. The maxima are exact: a cell left out lies below T, and T is below the
// speed of the cell that set it. Only the directions d < ndim (and the CFL rate when
// asked for) take part.

template <int PHYS, int NV>
__global__ void __launch_bounds__(256) speeds_kernel(SpeedParams p) {
  __shared__ unsigned long long red[4][32];
  __shared__ float redf[4][32];
  __shared__ float thr[4], thr_up[4];
  const int nitems = p.nitems_dev ? *p.nitems_dev : p.nitems;
  const float gam = (float)p.gamma;
  const bool want_rate = p.want_rate != 0;
  bool on[4];
#pragma unroll
  for (int q = 0; q < 4; q++) on[q] = q < 3 ? q < p.ndim : want_rate;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const CellItem ci = p.items[p.item0 + it];
    AMRFD_GUARD(p.err, cell_item_ok(p.doms, p.ndom, ci), continue)
    const DomDev dm = load_dom(p.doms + ci.dom);
    if (!p.active[dm.block0 + ci.blk]) continue;
    int o[3];
    block_coords(dm, ci.blk, o);
    const float rdx[3] = {(float)(1.0 / dm.dx[0]), (float)(1.0 / dm.dx[1]), (float)(1.0 / dm.dx[2])};
    unsigned* tl = p.tlow + (size_t)ci.dom * 4;
    float* iu = p.item_up ? p.item_up + (size_t)(p.item0 + it) * 4 : nullptr;
    float T[4] = {0.f, 0.f, 0.f, 0.f};
    if (p.exact) {
#pragma unroll
      for (int q = 0; q < 4; q++) T[q] = __uint_as_float(tl[q]);
      if (iu) {  // the same decision in every thread of the block
        bool any = false;
#pragma unroll
        for (int q = 0; q < 4; q++) any |= on[q] && iu[q] >= T[q];
        if (!any) continue;
      }
    }
    unsigned long long mx[4] = {0ull, 0ull, 0ull, 0ull};
    float lom[4] = {0.f, 0.f, 0.f, 0.f};
    float upm[4] = {0.f, 0.f, 0.f, 0.f};
    for (int c = threadIdx.x; c < ci.cnt; c += blockDim.x) {
      const int l = ci.c0 + c;
      const int lx = l % dm.be[0], ly = (l / dm.be[0]) % dm.be[1], lz = l / (dm.be[0] * dm.be[1]);
      const long long idx = dm.off + ((long long)(o[2] + lz) * dm.n[1] + (o[1] + ly)) * dm.n[0] + (o[0] + lx);
      double u[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) u[v] = p.U[idx + (long long)v * dm.ncell];
      if (p.W) {
        constexpr int NW = NumW<PHYS, NV>::value;
        double w[NW];
        prim_w<PHYS, NV>(u, p.gm1, w);
        const long long wi = dm.woff + (idx - dm.off);
#pragma unroll
        for (int q = 0; q < NW; q++) p.W[wi + (long long)q * dm.ncell] = w[q];
      }
      float up[4], lo[4];
      bool force;
      speed_bounds<PHYS, NV>(u, gam, p.ndim, rdx, want_rate, up, lo, force);
      if (!p.exact) {
        if (!force) {
#pragma unroll
          for (int q = 0; q < 4; q++) {
            lom[q] = fmaxf(lom[q], lo[q]);
            upm[q] = fmaxf(upm[q], up[q]);
          }
        } else {
#pragma unroll
          for (int q = 0; q < 4; q++) upm[q] = __int_as_float(0x7f800000);  // +inf
        }
        continue;
      }
      bool cand = force;
#pragma unroll
      for (int q = 0; q < 4; q++) cand |= on[q] && up[q] >= T[q];
      if (!cand) continue;
      if (!exact_speeds<PHYS, NV>(u, p.gamma, p.ndim, dm.dx, want_rate, mx)) atomicOr(p.err, kErrNonphysical);
    }
    if (!p.exact) {
      block_max4f_bcast(lom, redf, thr);
      if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < 4; q++)
          if (thr[q] > 0.f) atomicMax(tl + q, __float_as_uint(thr[q]));
      if (iu) {
        block_max4f_bcast(upm, redf, thr_up);
        if (threadIdx.x == 0)
#pragma unroll
          for (int q = 0; q < 4; q++) iu[q] = thr_up[q];
      }
      continue;
    }
    block_max4(mx, red);
    if (threadIdx.x == 0) {
#pragma unroll
      for (int q = 0; q < 4; q++)
        if (mx[q]) atomicMax(p.slot + (size_t)ci.dom * 4 + q, mx[q]);
    }
  }
}

// -------------------------------------------------------------------- flux
__device__ __forceinline__ double glm_speed(const unsigned long long* s0, int ndim) {
  double ch = 0.0;
  for (int d = 0; d < ndim; d++) ch = imax(ch, bitsd((long long)s0[d]));
  return ch;
}

// Splitting speed of an item's direction (raised to c_h with GLM) and c_h^2.
template <int D>
__device__ __forceinline__ double item_alpha(const FluxParams& p, const FluxItem& it, double& ch2) {
  const unsigned long long* sk = p.araw + (size_t)it.dom * 4;
  const unsigned long long* s0 = p.araw0 + (size_t)it.dom * 4;
  const double ch = p.glm ? glm_speed(s0, p.ndim) : 0.0;
  ch2 = ch * ch;
  return imax(bitsd((long long)sk[D]), ch);
}

// The cell whose values stand at coordinate g along dimension d (g may lie up to three cells
// outside): periodic wrap, the edge cell (zero gradient) or the mirror image; odd: the
// variables a mirror negates.
__device__ __forceinline__ int halo_cell(const DomDev& dm, int d, int g, unsigned& odd) {
  const int n = dm.n[d];
  odd = 0u;
  if (g < 0) {
    const int b = dm.bc[d][0];
    odd = dm.asym[d][0];
    return b == 0 ? g + n : (b == 1 ? 0 : -1 - g);
  }
  if (g >= n) {
    const int b = dm.bc[d][1];
    odd = dm.asym[d][1];
    return b == 0 ? g - n : (b == 1 ? n - 1 : 2 * n - 1 - g);
  }
  return g;
}

// Phase A of a flux item along D: the tile's G^{+-} (lines x segment + halo) into shared
// memory. FP64-bound: 33 of its ~150 instructions per cell, one per 64 cycles; the index
// arithmetic keeps no division and no block lookup in the loop (on the 1024^2 vortex the
// phase alone takes 0.152 ms of a launch, 87 % of it FP64 issue).
template <int PHYS, int NV, int D>
__device__ __forceinline__ void flux_phase_a(const FluxParams& p, const DomDev& dm, const FluxItem& it, double* sm) {
  constexpr int od1 = D == 0 ? 1 : 0;
  constexpr int od2 = D == 2 ? 1 : 2;
  const int W = it.slen + 2 * kGhost;
  const int nl = it.nl;
  const int P = nl, SS = tile_stride(it.slen);
  double ch2;
  const double alpha = item_alpha<D>(p, it, ch2);
  const double gm1 = p.gm1, one = ldk(K_ONE), mz = ldk(K_MZ);
  const int sx[3] = {1, dm.n[0], dm.n[0] * dm.n[1]};
  int o[3];
  block_coords(dm, it.blk, o);
  const int e1 = dm.be[od1];
  const int l1 = it.l0 % e1, l2 = it.l0 / e1;  // the first line
  const int g0 = o[D] + it.s0 - kGhost;
  const bool live = (it.live & kLiveHalo) != 0;
  // cells threadIdx.x, threadIdx.x + blockDim.x, ... of the tile, neighbouring threads along x
  const int inner = D == 0 ? W : nl, outer = D == 0 ? nl : W;
  int ou = threadIdx.x / inner, in = threadIdx.x - ou * inner;
  const int dou = blockDim.x / inner, din = blockDim.x - dou * inner;
  for (; ou < outer; ou += dou, in += din) {
    if (in >= inner) {
      in -= inner;
      if (++ou >= outer) break;
    }
    const int pl = D == 0 ? ou : in, j = D == 0 ? in : ou;
    int a1 = l1 + pl, a2 = l2;
    while (a1 >= e1) { a1 -= e1; a2++; }
    unsigned odd;
    const int g = halo_cell(dm, D, g0 + j, odd);
    const int x1 = o[od1] + a1, x2 = o[od2] + a2;
    AMRFD_GUARD(p.err, g >= 0 && g < dm.n[D] && x1 < dm.n[od1] && x2 < dm.n[od2] && pl < P && j < SS, continue)
    const long long idx = (long long)x1 * sx[od1] + (long long)x2 * sx[od2] + (long long)g * sx[D];
    bool act = true;
    if (!live) {  // a passive block is near: its cells are read as U^n
      int x[3];
      x[od1] = x1; x[od2] = x2; x[D] = g;
      act = p.active[dm.block0 + ((x[2] / dm.be[2]) * dm.nb[1] + x[1] / dm.be[1]) * dm.nb[0] + x[0] / dm.be[0]] != 0;
    }
    const double* src = (act ? p.Uk : p.Un) + dm.off + idx;
    constexpr int NW = NumW<PHYS, NV>::value;
    double u[NV], w[NW], gp[NV], gmn[NV];
#pragma unroll
    for (int v = 0; v < NV; v++) u[v] = src[(long long)v * dm.ncell];
    if (odd) {
#pragma unroll
      for (int v = 0; v < NV; v++)
        if ((odd >> v) & 1u) u[v] = dneg(u[v]);
    }
    // derived quantities: stored by the pass that produced U^(k) for active cells;
    // recomputed for passive neighbours (U^n) and mirror images
    if (p.W && act && !odd) {
      const double* ws = p.W + dm.woff + idx;
#pragma unroll
      for (int q = 0; q < NW; q++) w[q] = ws[(long long)q * dm.ncell];
    } else {
      prim_w<PHYS, NV>(u, gm1, w);
    }
    split_flux_w<PHYS, NV, D>(u, w, alpha, ch2, one, mz, gp, gmn);
#pragma unroll
    for (int v = 0; v < NV; v++) {
      sm[((0 * NV + v) * P + pl) * SS + j] = gp[v];
      sm[((1 * NV + v) * P + pl) * SS + j] = gmn[v];
    }
  }
}

// The variable whose MP5 sweeps cost clearly most and into how many times the parts it is
// worth sweeping it (1, 2 or 4), from the CTA's decaying per-variable counts of limiter
// faces per full part (cost[v], four times the recent average).
template <int NV>
__device__ __forceinline__ int hot_variable(const unsigned* cost, int plen, int& split) {
  int h = 0;
  unsigned m1 = 0u, m2 = 0u;
#pragma unroll
  for (int v = 0; v < NV; v++) {
    const unsigned c = cost[v];
    if (c > m1) { m2 = m1; m1 = c; h = v; }
    else if (c > m2) m2 = c;
  }
  split = m1 < (unsigned)plen || m1 < 2u * m2 ? 1 : (m1 < 2u * (unsigned)plen ? 2 : 4);
  return h;
}

// Phase B of a flux item: one thread per (variable, part, line) sweeps the part's faces
// and stores 60 times the flux difference of its cells (fixed_sweep; MODE 0: MP5; 1: MP5
// recording the limiter pieces; 2: LIMO3; 3: LIMO3 recording its pieces). The loop runs
// warp by warp: every lane of a warp takes the same number of trips, so that the sweeps'
// votes see exactly the lanes holding work.
// Balance (MP5): a face at which the limiter is needed costs about three times another
// face, so a variable limited at most of its faces (noise, a contact) would keep the CTA's
// other warps waiting at the barrier. Where the CTA has the threads, that variable
// (hot_variable, from the CTA's earlier items) is swept in two or four times as many parts.
// A face's value does not depend on the part that computes it.
template <int NV, int MODE>
__device__ __forceinline__ void flux_phase_b(const FluxParams& p, const DomDev& dm, const FluxItem& it,
                                             const double* sm, const unsigned* cost, unsigned* cost_new) {
  constexpr bool REC = MODE == 1 || MODE == 3;
  constexpr bool LIMO = MODE >= 2;
  const int d = it.d;
  const int nl = it.nl, slen = it.slen;
  const int np = sweep_parts(slen, p.part), P = nl, SS = tile_stride(slen);
  const int n = dm.n[d], be = dm.be[d];
  int o[3];
  block_coords(dm, it.blk, o);
  const int bstride = d == 0 ? 1 : (d == 1 ? dm.nb[0] : dm.nb[0] * dm.nb[1]);
  const int ostr = d == 0 ? 1 : (d == 1 ? dm.n[0] : dm.n[0] * dm.n[1]);
  const int od = d == 0 ? o[0] : (d == 1 ? o[1] : o[2]);
  const int f0 = od + it.s0;
  const unsigned char* row = p.active + dm.block0 + it.blk - (od / be) * bstride;  // blocks along the sweep
  // faces the segment's sweeps record (REC): those it owns, f0 .. f0 + slen - 1, and the
  // face after it where no segment owning that face runs: at an outflow or mirror end of
  // the line, or before a passive block (whose segments the forward pass skips; the
  // adjoint reads the face there). On a periodic line face n is face 0.
  int fend = f0 + slen;
  if constexpr (REC) {
    const bool at_end = fend == n;
    if (at_end && dm.bc[d][1] != 0) fend++;
    else if (!row[((at_end ? 0 : fend) / be) * bstride]) fend++;
  }
  const int fmod = dm.bc[d][1] == 0 ? n : n + 1;
  // cells of the segment inside active blocks (a segment through several blocks may
  // cross a passive one; every line of the item crosses the same blocks)
  unsigned long long wmask = slen >= 64 ? ~0ull : ((1ull << slen) - 1ull);
  if (!(it.live & kLiveAll)) {
    for (int j = 0; j < slen; j++)
      if (!row[((f0 + j) / be) * bstride]) wmask &= ~(1ull << j);
  }
  // the two dimensions across the lines
  const int e1 = d == 0 ? dm.be[1] : dm.be[0];
  const int s1 = d == 0 ? dm.n[0] : 1, s2 = d == 2 ? dm.n[0] : dm.n[0] * dm.n[1];
  const int l1 = it.l0 % e1, l2 = it.l0 / e1;
  const int o1 = d == 0 ? o[1] : o[0], o2 = d == 2 ? o[1] : o[2];
  double* Ld = p.L[d] + dm.off;
  const int nh = nl * np;
  int hot = 0, split = 1;
  if (!LIMO) {
    hot = hot_variable<NV>(cost, slen / np, split);
    while (split > 1 && (nh * split % 32 || slen / (np * split) < 4 || nh * (NV - 1 + split) > (int)blockDim.x))
      split >>= 1;
  }
  const int nhot = split > 1 ? nh * split : 0, total = nh * (NV - (nhot > 0)) + nhot;
  const int lane = threadIdx.x & 31;
  const double rdx = p.limo3_r * dm.dx[d];
  for (int t0 = threadIdx.x - lane; t0 < total; t0 += blockDim.x) {
    const int t = t0 + lane;
    const bool valid = t < total;
    const unsigned vm = __ballot_sync(0xffffffffu, valid);
    if (!valid) continue;
    // lines within parts within variables, the hot variable's parts first
    int v, r, parts = np;
    if (t < nhot) {
      v = hot;
      r = t;
      parts *= split;
    } else {
      v = (t - nhot) / nh;
      r = t - nhot - v * nh;
      if (nhot) v += v >= hot;
    }
    const int q = r / nl, pl = r - q * nl;
    const int p0 = q * slen / parts, len = (q + 1) * slen / parts - p0;
    const double* g = sm + (v * P + pl) * SS + p0;
    int a1 = l1 + pl, a2 = l2;
    while (a1 >= e1) { a1 -= e1; a2++; }
    const int x1 = o1 + a1, x2 = o2 + a2;
    double* out = Ld + (long long)v * dm.ncell + (long long)x1 * s1 + (long long)x2 * s2 + (long long)(f0 + p0) * ostr;
    const unsigned long long pmask = (wmask >> p0) & (len >= 64 ? ~0ull : ((1ull << len) - 1ull));
    unsigned short *tp = nullptr, *tm = nullptr;
    if constexpr (REC) {
      const int n1 = d == 0 ? dm.n[1] : dm.n[0], n2 = d == 2 ? dm.n[1] : dm.n[2];
      const long long ld = (long long)x2 * n1 + x1;
      tp = p.tape + dm.tape_off[d] + ((long long)(v * 2) * n1 * n2 + ld) * (n + 1);
      tm = tp + (long long)n1 * n2 * (n + 1);
    }
    // a part records the faces it owns: its left face and interior faces; the
    // segment's last part also the faces the segment owns at its right end
    const int fe = p0 + len == slen ? fend : f0 + p0 + len;
    const line_t gl = (line_t)__cvta_generic_to_shared(g);
    const int limited = fixed_sweep<LIMO, REC>(gl, line_at(gl, NV * P * SS), len, 4.0 * rdx * rdx, out, ostr, pmask,
                                               tp, tm, f0 + p0, fe, fmod, vm);
    if (!LIMO && limited) atomicMax(cost_new + v, (unsigned)(limited * (parts / np)));
  }
}

template <int PHYS, int NV, int MODE>
__global__ void __launch_bounds__(kFluxMaxThreads, 2) flux_kernel(FluxParams p) {
  extern __shared__ double sm[];
  __shared__ int s_it;
  __shared__ unsigned s_cost[32];  // limiter faces per variable: decaying sum, this item's
  if (threadIdx.x < 32) s_cost[threadIdx.x] = 0u;
  __syncthreads();
  const int nitems = p.nitems_dev ? *p.nitems_dev : p.nitems;
  int it;
  if (p.counter) {
    if (threadIdx.x == 0) s_it = atomicAdd(p.counter, 1);
    __syncthreads();
    it = s_it;
    __syncthreads();
  } else {
    it = blockIdx.x;
  }
  constexpr int maxd = PHYS == PH_EULER ? NV - 2 : 3;
  while (it < nitems) {
    const FluxItem item = p.items[p.item0 + it];
    bool live = (item.live & kLiveAny) != 0;
    AMRFD_GUARD(p.err, flux_item_ok(p.doms, p.ndom, p.ndim, p.P, p.SS, item), live = false)
    if (live) {  // phase A, barrier, phase B, barrier
      const DomDev& dm = p.doms[item.dom];
      if (threadIdx.x < NV) {  // the last item's counts were added before its last barrier
        const unsigned c = s_cost[threadIdx.x];
        s_cost[threadIdx.x] = c - (c >> 2) + s_cost[16 + threadIdx.x];
        s_cost[16 + threadIdx.x] = 0u;
      }
      if (item.d == 0) flux_phase_a<PHYS, NV, 0>(p, dm, item, sm);
      if constexpr (maxd > 1) { if (item.d == 1) flux_phase_a<PHYS, NV, (maxd > 1 ? 1 : 0)>(p, dm, item, sm); }
      if constexpr (maxd > 2) { if (item.d == 2) flux_phase_a<PHYS, NV, (maxd > 2 ? 2 : 0)>(p, dm, item, sm); }
      __syncthreads();
      flux_phase_b<NV, MODE>(p, dm, item, sm, s_cost, s_cost + 16);
      __syncthreads();
    }
    if (p.counter) {
      if (threadIdx.x == 0) s_it = atomicAdd(p.counter, 1);
      __syncthreads();
      it = s_it;
      __syncthreads();
    } else {
      it += gridDim.x;
    }
  }
}

// ----------------------------------------------------------------- combine
// The derived quantities and FP32 speed bounds of one new state u (cell at idx).
template <int PHYS, int NV>
__device__ __forceinline__ void combine_tail(const CombParams& p, const DomDev& dm, long long idx, const double* u,
                                             float gam, float lom[4], float upm[4]) {
  const float rdx[3] = {0.f, 0.f, 0.f};
  if (p.W) {
    constexpr int NW = NumW<PHYS, NV>::value;
    double w[NW];
    prim_w<PHYS, NV>(u, p.gm1, w);
    const long long wi = dm.woff + (idx - dm.off);
#pragma unroll
    for (int q = 0; q < NW; q++) p.W[wi + (long long)q * dm.ncell] = w[q];
  }
  if (p.tlow_out) {
    float up[4], lo[4];
    bool force;
    speed_bounds<PHYS, NV>(u, gam, p.ndim, rdx, false, up, lo, force);
    if (!force) {
#pragma unroll
      for (int q = 0; q < 3; q++) {
        lom[q] = fmaxf(lom[q], lo[q]);
        upm[q] = fmaxf(upm[q], up[q]);
      }
    } else {
#pragma unroll
      for (int q = 0; q < 3; q++) upm[q] = __int_as_float(0x7f800000);  // +inf
    }
  }
}

// The cells of one item. Every load of a cell is issued before its stores (the output
// may be the U^n buffer, so loads cannot move past a store); A0ONE skips the product
// with a first coefficient of 1. Per variable the operations and their order are
// a_0 U^(k_0), then a_t U^(k_t) and w_d L_d by FMA, then the psi damping.
template <int PHYS, int NV, bool A0ONE>
__device__ __forceinline__ void combine_cells(const CombParams& p, const DomDev& dm, const CellItem& ci,
                                              const int o[3], double w0, double w1, double w2, double fac,
                                              float gam, float lom[4], float upm[4]) {
  const long long nc = dm.ncell;
  for (int c = threadIdx.x; c < ci.cnt; c += blockDim.x) {
    const int l = ci.c0 + c;
    const int lx = l % dm.be[0], ly = (l / dm.be[0]) % dm.be[1], lz = l / (dm.be[0] * dm.be[1]);
    const long long idx = dm.off + ((long long)(o[2] + lz) * dm.n[1] + (o[1] + ly)) * dm.n[0] + (o[0] + lx);
    double u[NV];
    {
      const double* b0 = p.buf[p.co.k[0]] + idx;
#pragma unroll
      for (int v = 0; v < NV; v++) u[v] = A0ONE ? b0[v * nc] : p.co.a[0] * b0[v * nc];
    }
    for (int t = 1; t < p.co.nterm; t++) {
      const double* bt = p.buf[p.co.k[t]] + idx;
      const double at = p.co.a[t];
#pragma unroll
      for (int v = 0; v < NV; v++) u[v] = fma(at, bt[v * nc], u[v]);
    }
    {
      const double* L0 = p.L[0] + idx;
#pragma unroll
      for (int v = 0; v < NV; v++) u[v] = fma(w0, L0[v * nc], u[v]);
    }
    if (p.ndim > 1) {
      const double* L1 = p.L[1] + idx;
#pragma unroll
      for (int v = 0; v < NV; v++) u[v] = fma(w1, L1[v * nc], u[v]);
    }
    if (p.ndim > 2) {
      const double* L2 = p.L[2] + idx;
#pragma unroll
      for (int v = 0; v < NV; v++) u[v] = fma(w2, L2[v * nc], u[v]);
    }
    if constexpr (PHYS == PH_MHD) u[NV - 1] *= fac;  // psi
#pragma unroll
    for (int v = 0; v < NV; v++) p.out[idx + v * nc] = u[v];
    combine_tail<PHYS, NV>(p, dm, idx, u, gam, lom, upm);
  }
}

// combine_cells for two neighbouring cells along x per thread, read and written with
// 16-byte (double2) accesses; the same operations in the same order on each cell. The
// caller checks that every pair starts 16-byte aligned.
template <int PHYS, int NV, bool A0ONE>
__device__ __forceinline__ void combine_pairs(const CombParams& p, const DomDev& dm, const CellItem& ci,
                                              const int o[3], double w0, double w1, double w2, double fac,
                                              float gam, float lom[4], float upm[4]) {
  const long long nc = dm.ncell;
  for (int c = threadIdx.x; c < ci.cnt / 2; c += blockDim.x) {
    const int l = ci.c0 + 2 * c;
    const int lx = l % dm.be[0], ly = (l / dm.be[0]) % dm.be[1], lz = l / (dm.be[0] * dm.be[1]);
    const long long idx = dm.off + ((long long)(o[2] + lz) * dm.n[1] + (o[1] + ly)) * dm.n[0] + (o[0] + lx);
    double ua[NV], ub[NV];
    {
      const double* b0 = p.buf[p.co.k[0]] + idx;
#pragma unroll
      for (int v = 0; v < NV; v++) {
        const double2 x = *reinterpret_cast<const double2*>(b0 + v * nc);
        ua[v] = A0ONE ? x.x : p.co.a[0] * x.x;
        ub[v] = A0ONE ? x.y : p.co.a[0] * x.y;
      }
    }
    for (int t = 1; t < p.co.nterm; t++) {
      const double* bt = p.buf[p.co.k[t]] + idx;
      const double at = p.co.a[t];
#pragma unroll
      for (int v = 0; v < NV; v++) {
        const double2 x = *reinterpret_cast<const double2*>(bt + v * nc);
        ua[v] = fma(at, x.x, ua[v]);
        ub[v] = fma(at, x.y, ub[v]);
      }
    }
    for (int d = 0; d < p.ndim; d++) {
      const double* Ld = p.L[d] + idx;
      const double wd = d == 0 ? w0 : (d == 1 ? w1 : w2);
#pragma unroll
      for (int v = 0; v < NV; v++) {
        const double2 x = *reinterpret_cast<const double2*>(Ld + v * nc);
        ua[v] = fma(wd, x.x, ua[v]);
        ub[v] = fma(wd, x.y, ub[v]);
      }
    }
    if constexpr (PHYS == PH_MHD) {
      ua[NV - 1] *= fac;  // psi
      ub[NV - 1] *= fac;
    }
#pragma unroll
    for (int v = 0; v < NV; v++) *reinterpret_cast<double2*>(p.out + idx + v * nc) = make_double2(ua[v], ub[v]);
    for (int half = 0; half < 2; half++) combine_tail<PHYS, NV>(p, dm, idx + half, half ? ub : ua, gam, lom, upm);
  }
}

template <int PHYS, int NV>
__global__ void __launch_bounds__(256) combine_kernel(CombParams p) {
  __shared__ float redf[4][32];
  __shared__ float thr[4], thr_up[4];
  __shared__ double s_fac;
  const int nitems = p.nitems_dev ? *p.nitems_dev : p.nitems;
  const float gam = (float)p.gamma;
  const bool a0_one = p.co.a[0] == 1.0;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const CellItem ci = p.items[p.item0 + it];
    AMRFD_GUARD(p.err, cell_item_ok(p.doms, p.ndom, ci), continue)
    const DomDev dm = load_dom(p.doms + ci.dom);
    if (!p.active[dm.block0 + ci.blk]) continue;
    int o[3];
    block_coords(dm, ci.blk, o);
    const double dt = p.dt[ci.dom];
    const double dtb = dt * p.co.b;
    // L = sum_d (Fsum_{i-1/2} - Fsum_{i+1/2}) / (2 dx_d), Fsum in units of 2 F^; the flux pass
    // stores 60 times the differences
    const double w0 = stage_weight(dtb, dm.dx[0]);
    const double w1 = p.ndim > 1 ? stage_weight(dtb, dm.dx[1]) : 0.0;
    const double w2 = p.ndim > 2 ? stage_weight(dtb, dm.dx[2]) : 0.0;
    const bool damp = PHYS == PH_MHD && p.final_stage && p.glm_cr > 0.0;
    if (damp) {
      if (threadIdx.x == 0) {
        const double ch = glm_speed(p.araw0 + (size_t)ci.dom * 4, p.ndim);
        s_fac = exp(-dt * ch / p.glm_cr);
      }
      __syncthreads();
    }
    const double fac = damp ? s_fac : 1.0;
    float lom[4] = {0.f, 0.f, 0.f, 0.f};
    float upm[4] = {0.f, 0.f, 0.f, 0.f};
    // pairs along x when every pair starts 16-byte aligned: buffers aligned (host), an even
    // x extent and block edge, an even domain offset and item start and count
    const bool pair = p.pairs && !((dm.n[0] | dm.be[0] | ci.c0 | ci.cnt) & 1) && !(dm.off & 1);
    if (pair) {
      if (a0_one) combine_pairs<PHYS, NV, true>(p, dm, ci, o, w0, w1, w2, fac, gam, lom, upm);
      else combine_pairs<PHYS, NV, false>(p, dm, ci, o, w0, w1, w2, fac, gam, lom, upm);
    } else {
      if (a0_one) combine_cells<PHYS, NV, true>(p, dm, ci, o, w0, w1, w2, fac, gam, lom, upm);
      else combine_cells<PHYS, NV, false>(p, dm, ci, o, w0, w1, w2, fac, gam, lom, upm);
    }
    if (p.tlow_out) {
      block_max4f_bcast(lom, redf, thr);
      if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < 3; q++)
          if (thr[q] > 0.f) atomicMax(p.tlow_out + (size_t)ci.dom * 4 + q, __float_as_uint(thr[q]));
      if (p.item_up) {
        block_max4f_bcast(upm, redf, thr_up);
        if (threadIdx.x == 0)
#pragma unroll
          for (int q = 0; q < 4; q++) p.item_up[(size_t)(p.item0 + it) * 4 + q] = thr_up[q];
      }
    } else if (damp) {
      __syncthreads();  // s_fac is rewritten by the next item
    }
  }
}

// --------------------------------------------------------------------- dt
__global__ void __launch_bounds__(1024) dt_kernel(DtParams p) {
  __shared__ long long red[32];
  long long best = 0x7fffffffffffffffLL;  // okey of the minimum over this thread's domains
  for (int dmi = threadIdx.x; dmi < p.ndom; dmi += blockDim.x) {
    const DomDev& dm = p.doms[dmi];
    const unsigned long long* s = p.slot + (size_t)dmi * 4;
    double rate;
    if (p.glm) {
      double ch = 0.0;
      for (int d = 0; d < p.ndim; d++) ch = imax(ch, bitsd((long long)s[d]));
      rate = 0.0;
      for (int d = 0; d < p.ndim; d++) rate = __dadd_rn(rate, __ddiv_rn(ch, dm.dx[d]));
    } else {
      rate = bitsd((long long)s[3]);
    }
    double dt = rate > 0.0 ? __ddiv_rn(p.cfl, rate) : __longlong_as_double(0x7ff0000000000000LL);
    const double rem = __dsub_rn(p.t_end, p.t);
    dt = imin(dt, rem);
    p.dt_out[dmi] = dt;
    const long long k = okey(dt);
    best = k < best ? k : best;
  }
  if (!p.global_min) return;
  for (int o = 16; o > 0; o >>= 1) {
    long long y = __shfl_xor_sync(0xffffffffu, best, o);
    best = y < best ? y : best;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x < 32) {
    long long x = threadIdx.x < (blockDim.x + 31) / 32 ? red[threadIdx.x] : 0x7fffffffffffffffLL;
    for (int o = 16; o > 0; o >>= 1) {
      long long y = __shfl_xor_sync(0xffffffffu, x, o);
      x = y < x ? y : x;
    }
    if (threadIdx.x == 0) red[0] = x;
  }
  __syncthreads();
  const long long kb = red[0];
  const double dmin = bitsd(kb ^ ((kb >> 63) & 0x7fffffffffffffffLL));
  for (int dmi = threadIdx.x; dmi < p.ndom; dmi += blockDim.x) p.dt_out[dmi] = dmin;
}

// ------------------------------------------------------------- compaction
__device__ __forceinline__ bool group_live(const CompactParams& p, int i) {
  const int o = p.list.owner[i], st = p.list.stride[i], sp = p.list.span[i];
  bool live = false;
  for (int m = 0; m < sp; m++) live |= p.active[o + m * st] != 0;
  return live;
}

__global__ void __launch_bounds__(1024) compact_scan_kernel(CompactParams p) {
  __shared__ int wsum[32];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int base = 0; base < p.list.ngroups; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const int f = (i < p.list.ngroups && group_live(p, i)) ? p.list.cnt[i] : 0;
    int fs = f;
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, fs, o);
      if (lane >= o) fs += a;
    }
    if (lane == 31) wsum[wid] = fs;
    __syncthreads();
    if (wid == 0) {
      const int nw = blockDim.x >> 5;
      int a = lane < nw ? wsum[lane] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, a, o);
        if (lane >= o) a += x;
      }
      if (lane < nw) wsum[lane] = a;
    }
    __syncthreads();
    const int fo = carry + (wid ? wsum[wid - 1] : 0) + fs - f;
    if (i < p.list.ngroups) p.list.dst[i] = f ? fo : -1;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = fo + f;
    __syncthreads();
  }
  if (threadIdx.x == 0) *p.list.count = carry;
}

// ItemLive bits of a flux item.
__device__ __forceinline__ unsigned char item_liveness(const CompactParams& p, const FluxItem& item) {
  const DomDev& dm = p.doms[item.dom];
  const int d = item.d, be = dm.be[d];
  const int bstride = d == 0 ? 1 : (d == 1 ? dm.nb[0] : dm.nb[0] * dm.nb[1]);
  int o[3];
  block_coords(dm, item.blk, o);
  const int od = d == 0 ? o[0] : (d == 1 ? o[1] : o[2]);
  const unsigned char* row = p.active + dm.block0 + item.blk - (od / be) * bstride;
  const int c0 = od + item.s0, c1 = c0 + item.slen;
  bool any = false, all = true;
  for (int b = c0 / be; b <= (c1 - 1) / be; b++) {
    const bool a = row[b * bstride] != 0;
    any |= a;
    all &= a;
  }
  bool halo = all;
  for (int j = 1; j <= kGhost && halo; j++) {
    unsigned odd;
    halo = row[halo_cell(dm, d, c0 - j, odd) / be * bstride] && row[halo_cell(dm, d, c1 - 1 + j, odd) / be * bstride];
  }
  return (unsigned char)((any ? kLiveAny : 0) | (all ? kLiveAll : 0) | (halo ? kLiveHalo : 0));
}

// Copies the live groups' items; flux items of every group get their liveness bits first
// (the plain path runs through the full list).
__global__ void __launch_bounds__(256) compact_copy_kernel(CompactParams p) {
  const int w = p.list.item_bytes / 4;
  unsigned* in = (unsigned*)p.list.in;
  unsigned* out = (unsigned*)p.list.out;
  for (int i = blockIdx.x; i < p.list.ngroups; i += gridDim.x) {
    const int d = p.list.dst[i];
    const int b = p.list.beg[i], c = p.list.cnt[i];
    if (p.flux_items) {
      FluxItem* fi = (FluxItem*)p.list.in + b;
      for (int t = threadIdx.x; t < c; t += blockDim.x) fi[t].live = item_liveness(p, fi[t]);
      __syncthreads();
    }
    if (d < 0) continue;
    for (int t = threadIdx.x; t < c * w; t += blockDim.x) out[(size_t)d * w + t] = in[(size_t)b * w + t];
  }
}

// ------------------------------------------------------------- dispatch
#define AMRFD_DISPATCH(physics, nv, CALL)                                   \
  do {                                                                      \
    if ((physics) == PH_MHD && (nv) == 9) { CALL(PH_MHD, 9); }              \
    else if ((physics) == PH_EULER && (nv) == 3) { CALL(PH_EULER, 3); }     \
    else if ((physics) == PH_EULER && (nv) == 4) { CALL(PH_EULER, 4); }     \
    else if ((physics) == PH_EULER && (nv) == 5) { CALL(PH_EULER, 5); }     \
    else return cudaErrorInvalidValue;                                      \
  } while (0)

cudaError_t launch_speeds(int physics, int nv, const SpeedParams& p, int grid, int block, cudaStream_t s) {
#define CALL(PH, NVV) speeds_kernel<PH, NVV><<<grid, block, 0, s>>>(p)
  AMRFD_DISPATCH(physics, nv, CALL);
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_flux(int physics, int nv, const FluxParams& p, int grid, int block, size_t smem, cudaStream_t s) {
#define CALL(PH, NVV)                                                                \
  if (p.tape && p.limo3) flux_kernel<PH, NVV, 3><<<grid, block, smem, s>>>(p);      \
  else if (p.tape) flux_kernel<PH, NVV, 1><<<grid, block, smem, s>>>(p);            \
  else if (p.limo3) flux_kernel<PH, NVV, 2><<<grid, block, smem, s>>>(p);           \
  else flux_kernel<PH, NVV, 0><<<grid, block, smem, s>>>(p)
  AMRFD_DISPATCH(physics, nv, CALL);
#undef CALL
  return cudaGetLastError();
}

// Lets a kernel take all the dynamic shared memory a block may have. The attribute belongs
// to the function, not to a handle or a launch: set to one handle's tile it would refuse
// another handle's larger one.
cudaError_t allow_smem(const void* fn) {
  cudaFuncAttributes at;
  cudaError_t e = cudaFuncGetAttributes(&at, fn);
  int dev = 0, most = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)at.sharedSizeBytes);
}

cudaError_t flux_allow_smem(int physics, int nv) {
#define CALL(PH, NVV)                                                                               \
  for (const void* fn : {(const void*)flux_kernel<PH, NVV, 0>, (const void*)flux_kernel<PH, NVV, 1>, \
                         (const void*)flux_kernel<PH, NVV, 2>, (const void*)flux_kernel<PH, NVV, 3>}) { \
    cudaError_t e = allow_smem(fn);                                                                 \
    if (e != cudaSuccess) return e;                                                                 \
  }
  AMRFD_DISPATCH(physics, nv, CALL);
#undef CALL
  return cudaSuccess;
}

cudaError_t flux_occupancy(int physics, int nv, int limo3, int block, size_t smem, int* per_sm) {
#define CALL(PH, NVV)                                                                                        \
  return limo3 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, flux_kernel<PH, NVV, 2>, block, smem) \
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, flux_kernel<PH, NVV, 0>, block, smem)
  AMRFD_DISPATCH(physics, nv, CALL);
#undef CALL
  return cudaSuccess;
}

cudaError_t launch_combine(int physics, int nv, const CombParams& p, int grid, int block, cudaStream_t s) {
#define CALL(PH, NVV) combine_kernel<PH, NVV><<<grid, block, 0, s>>>(p)
  AMRFD_DISPATCH(physics, nv, CALL);
#undef CALL
  return cudaGetLastError();
}

// One round of App. C's safety belt: a candidate block becomes active when one of
// its (up to 26) neighbours was active in the previous round; neighbours wrap across
// periodic faces and do not exist beyond other faces. The first pass only inverts
// the candidate flags.
__global__ void activate_kernel(ActParams p) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < p.nblocks; b += gridDim.x * blockDim.x) {
    if (p.first) { p.out[b] = p.in[b] ? 0 : 1; continue; }
    unsigned char a = p.in[b];
    if (!a) {
      const DomDev& dm = p.doms[p.bdom[b]];
      const int l = b - dm.block0;
      const int i[3] = {l % dm.nb[0], (l / dm.nb[0]) % dm.nb[1], l / (dm.nb[0] * dm.nb[1])};
      int lo[3], hi[3];
#pragma unroll
      for (int k = 0; k < 3; k++) { lo[k] = dm.nb[k] > 1 ? -1 : 0; hi[k] = -lo[k]; }
      for (int oz = lo[2]; oz <= hi[2] && !a; oz++)
        for (int oy = lo[1]; oy <= hi[1] && !a; oy++)
          for (int ox = lo[0]; ox <= hi[0] && !a; ox++) {
            const int o[3] = {ox, oy, oz};
            int j[3];
            bool ok = true;
#pragma unroll
            for (int k = 0; k < 3; k++) {
              j[k] = i[k] + o[k];
              if (j[k] < 0 || j[k] >= dm.nb[k]) {
                if (dm.bc[k][0] == 0) j[k] = j[k] < 0 ? j[k] + dm.nb[k] : j[k] - dm.nb[k];
                else ok = false;
              }
            }
            if (ok && p.in[dm.block0 + (j[2] * dm.nb[1] + j[1]) * dm.nb[0] + j[0]]) a = 1;
          }
    }
    p.out[b] = a;
  }
}

// Steady-state criterion over cell items; flag[] was set to 1 beforehand. NaN counts as
// a deviation.
__global__ void __launch_bounds__(256) flag_steady_kernel(FlagParams p) {
  for (int it = blockIdx.x; it < p.nitems; it += gridDim.x) {
    const CellItem ci = p.items[it];
    AMRFD_GUARD(p.err, cell_item_ok(p.doms, p.ndom, ci), continue)
    const DomDev dm = load_dom(p.doms + ci.dom);
    int o[3];
    block_coords(dm, ci.blk, o);
    int dev = 0;
    for (int c = threadIdx.x; c < ci.cnt && !dev; c += blockDim.x) {
      const int l = ci.c0 + c;
      const int lx = l % dm.be[0], ly = (l / dm.be[0]) % dm.be[1], lz = l / (dm.be[0] * dm.be[1]);
      const long long idx = dm.off + ((long long)(o[2] + lz) * dm.n[1] + (o[1] + ly)) * dm.n[0] + (o[0] + lx);
      for (int v = 0; v < p.nv; v++) {
        const long long e = idx + (long long)v * dm.ncell;
        if (!(fabs(p.U[e] - p.R[e]) <= p.tol)) { dev = 1; break; }
      }
    }
    if (__syncthreads_or(dev) && threadIdx.x == 0) p.flag[dm.block0 + ci.blk] = 0;
  }
}

cudaError_t launch_activate(const ActParams& p, cudaStream_t s) {
  const int grid = p.nblocks > 0 ? (p.nblocks + 255) / 256 : 1;
  activate_kernel<<<grid < 1024 ? grid : 1024, 256, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_flag_steady(const FlagParams& p, int grid, cudaStream_t s) {
  flag_steady_kernel<<<grid, 256, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_dt(const DtParams& p, cudaStream_t s) {
  dt_kernel<<<1, 1024, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_compact(const CompactParams& p, cudaStream_t s) {
  compact_scan_kernel<<<1, 1024, 0, s>>>(p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int n = p.list.ngroups;
  compact_copy_kernel<<<n < 4096 ? (n > 0 ? n : 1) : 4096, 256, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace amrfd
