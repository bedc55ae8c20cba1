// amrfd_adjoint.cu -- discrete adjoint of one SSPRK step of the FD-MP5 update.
//
// With the splitting speeds c_max (per stage), the GLM speed c_h and the psi
// damping factor held at their forward values, one stage is
//   U^(i) = sum_t a_t U^(k_t) + sum_d w_d D_d(S),   S = U^(i-1), w_d = dt b / (2 dx_d),
// where D_d(S)_j = Fsum_j - Fsum_{j+1} and Fsum_k = G+_{k-1} + G-_k + (Y+_k + Y-_k)/2
// is the interface flux of Sec. 2.2 in units of 2 F^ (G = F +- c_max U). Every MP5
// value Y is piecewise linear in its stencil once the limiter's choices are fixed;
// the forward recomputation records, per face, variable and bias, which pieces the
// limiter took (a 9-bit tape), and the adjoint applies their transposes without
// re-evaluating the limiter. Gradients are gathered per cell (no atomics):
// a segment recomputes the faces within reach of its cells (two beyond on the low
// side, three on the high side) and keeps only contributions to its own cells;
// with outflow faces the ghost copies of an edge cell fold back into it.
#include <cuda_runtime.h>

#include "amrfd_device.cuh"
#include "amrfd_kernels.cuh"
#include "amrfd_sweep.cuh"

namespace amrfd {

// Transposed flux-split Jacobian: gu = (dG+/dU)^T gp + (dG-/dU)^T gm with
// G+- = F_D(U) +- alpha U (alpha, c_h fixed).
template <int PHYS, int NV, int D>
__device__ __forceinline__ void split_flux_adj(const double* u, double gm1, double alpha, double ch2,
                                               const double* gp, const double* gmn, double* gu) {
  double y[NV];
#pragma unroll
  for (int v = 0; v < NV; v++) {
    y[v] = gp[v] + gmn[v];
    gu[v] = alpha * (gp[v] - gmn[v]);
  }
  const double rho = u[0];
  const double ir = frcp(rho);
  if (PHYS == PH_EULER) {
    constexpr int nm = NV - 2;
    double v[nm], gv[nm];
    double mv = 0.0;
#pragma unroll
    for (int k = 0; k < nm; k++) { v[k] = u[1 + k] * ir; mv = fma(u[1 + k], v[k], mv); gv[k] = 0.0; }
    const double E = u[NV - 1];
    const double p = gm1 * fma(-0.5, mv, E);
    const double vd = v[D];
    double gp_ = 0.0, gE = 0.0;
    gu[1 + D] += y[0];
#pragma unroll
    for (int k = 0; k < nm; k++) {
      gv[D] += y[1 + k] * u[1 + k];
      gu[1 + k] += y[1 + k] * vd;
      if (k == D) gp_ += y[1 + k];
    }
    gv[D] += y[NV - 1] * (E + p);
    gE += y[NV - 1] * vd;
    gp_ += y[NV - 1] * vd;
    gE += gm1 * gp_;
    const double gmv = -0.5 * gm1 * gp_;
    double gir = 0.0;
#pragma unroll
    for (int k = 0; k < nm; k++) {
      gu[1 + k] += gmv * v[k];
      gv[k] += gmv * u[1 + k];
      gu[1 + k] += gv[k] * ir;
      gir += gv[k] * u[1 + k];
    }
    gu[0] -= gir * ir * ir;
    gu[NV - 1] += gE;
  } else {
    const double E = u[4];
    const double B[3] = {u[5], u[6], u[7]};
    const double v[3] = {u[1] * ir, u[2] * ir, u[3] * ir};
    const double b2 = fma(B[2], B[2], fma(B[1], B[1], B[0] * B[0]));
    const double mv = fma(u[3], v[2], fma(u[2], v[1], u[1] * v[0]));
    const double p = gm1 * fma(-0.5, mv + b2, E);
    const double ptot = fma(0.5, b2, p);
    const double vb = fma(v[2], B[2], fma(v[1], B[1], v[0] * B[0]));
    const double vd = v[D], bd = B[D];
    double gv[3] = {0.0, 0.0, 0.0}, gB[3] = {0.0, 0.0, 0.0};
    double gptot = 0.0, gE = 0.0, gvb = 0.0, gpsi = 0.0;
    gu[1 + D] += y[0];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const double yk = y[1 + k];
      gv[D] += yk * u[1 + k];
      gu[1 + k] += yk * vd;
      gB[D] -= yk * B[k];
      gB[k] -= yk * bd;
      if (k == D) gptot += yk;
    }
    gv[D] += y[4] * (E + ptot);
    gE += y[4] * vd;
    gptot += y[4] * vd;
    gB[D] -= y[4] * vb;
    gvb -= y[4] * bd;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const double yk = y[5 + k];
      if (k == D) {
        gpsi += yk;
      } else {
        gv[D] += yk * B[k];
        gB[k] += yk * vd;
        gB[D] -= yk * v[k];
        gv[k] -= yk * bd;
      }
    }
    gB[D] += y[8] * ch2;
#pragma unroll
    for (int k = 0; k < 3; k++) { gv[k] += gvb * B[k]; gB[k] += gvb * v[k]; }
    double gb2 = 0.5 * gptot;
    const double gp_ = gptot;
    gE += gm1 * gp_;
    const double gmv = -0.5 * gm1 * gp_;
    gb2 -= 0.5 * gm1 * gp_;
    double gir = 0.0;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      gu[1 + k] += gmv * v[k];
      gv[k] += gmv * u[1 + k];
      gB[k] += 2.0 * B[k] * gb2;
      gu[1 + k] += gv[k] * ir;
      gir += gv[k] * u[1 + k];
      gu[5 + k] += gB[k];
    }
    gu[0] -= gir * ir * ir;
    gu[4] += gE;
    gu[8] += gpsi;
  }
}

// Whether the block next to block `blk` along d (side -1 or +1) exists and is active
// (wrapping across periodic faces).
__device__ __forceinline__ bool nb_active(const DomDev& dm, const unsigned char* active, int blk, int d, int side) {
  const int bi[3] = {blk % dm.nb[0], (blk / dm.nb[0]) % dm.nb[1], blk / (dm.nb[0] * dm.nb[1])};
  int j = bi[d] + side;
  if (j < 0 || j >= dm.nb[d]) {
    if (dm.bc[d][0] != 0) return false;
    j = j < 0 ? j + dm.nb[d] : j - dm.nb[d];
  }
  const int stride = d == 0 ? 1 : (d == 1 ? dm.nb[0] : dm.nb[0] * dm.nb[1]);
  return active[dm.block0 + blk + (j - bi[d]) * stride] != 0;
}

// A passive block whose cells fed an active neighbour's fluxes along d: the active cells'
// faces reach three cells into it (blocks hold at least three cells along d when their
// domain is partly active), where the forward pass read U^n.
__device__ __forceinline__ bool passive_fed(const DomDev& dm, const unsigned char* active, int blk, int d) {
  return !active[dm.block0 + blk] && (nb_active(dm, active, blk, d, -1) || nb_active(dm, active, blk, d, 1));
}

template <int PHYS, int NV, int D, bool LIMO>
__device__ __forceinline__ void adj_item(const AdjFluxParams& p, const FluxItem& it, double* sm) {
  constexpr int od1 = D == 0 ? 1 : 0;
  constexpr int od2 = D == 2 ? 1 : 2;
  const DomDev dm = *(p.doms + it.dom);
  int o[3];
  {
    const int bx = it.blk % dm.nb[0], by = (it.blk / dm.nb[0]) % dm.nb[1], bz = it.blk / (dm.nb[0] * dm.nb[1]);
    o[0] = bx * dm.be[0]; o[1] = by * dm.be[1]; o[2] = bz * dm.be[2];
  }
  const unsigned long long* sk = p.araw + (size_t)it.dom * 4;
  const unsigned long long* s0p = p.araw0 + (size_t)it.dom * 4;
  double ch = 0.0;
  if (p.glm)
    for (int d = 0; d < p.ndim; d++) ch = imax(ch, bitsd((long long)s0p[d]));
  const double alpha = imax(bitsd((long long)sk[D]), ch);
  const double ch2 = ch * ch;
  // the transposed sweeps give 60 times the gradient: w + wl = dt b / (120 dx) to twice the
  // precision, since the weight's rounding would bias every cell alike
  const double den = 120.0 * dm.dx[D], rden = 1.0 / den, num = p.dt[it.dom] * p.b;
  const double w = num * rden;
  const double wl = (fma(-w, den, num) + (fma(p.dt[it.dom], p.b, -num) - w * fma(120.0, dm.dx[D], -den))) * rden;
  const double pfac = p.psi_fac ? p.psi_fac[it.dom] : 1.0;
  const int nl = it.nl, slen = it.slen, P = p.P, SA = p.SSa, SG = p.SSg;
  const int n = dm.n[D];
  const int s0 = o[D] + it.s0;               // first cell of the segment (domain coordinate)
  const int WG = slen + 6;
  double* gGp = sm;                           // [NV][P][SA] gradient w.r.t. G+ at positions s0-5 ..
  double* gGm = gGp + NV * P * SA;
  double* gh = gGm + NV * P * SA;             // [NV][P][SG] scaled upstream gradient at s0-3 ..
  // passive block (fed an active neighbour): its cells entered the fluxes as U^n
  const bool self_active = p.active[dm.block0 + it.blk] != 0;
  const int bstride = D == 0 ? 1 : (D == 1 ? dm.nb[0] : dm.nb[0] * dm.nb[1]);
  const int bo = it.blk - (o[D] / dm.be[D]) * bstride;  // block index with coordinate D = 0
  // ---- phase A: upstream gradient at s0-3 .. s0+slen+2 (zero beyond an outflow face and
  // at passive cells, whose residual the step does not use)
  for (int c = threadIdx.x; c < nl * WG; c += blockDim.x) {
    int pl, r;
    if (D == 0) { pl = c / WG; r = c - pl * WG; }
    else { r = c / nl; pl = c - r * nl; }
    const int line = it.l0 + pl;
    const int a1 = line % dm.be[od1], a2 = line / dm.be[od1];
    int x[3];
    x[od1] = o[od1] + a1;
    x[od2] = o[od2] + a2;
    int g = s0 - 3 + r;
    bool live = true;
    if (g < 0) { live = dm.bc[D][0] == 0; g = ((g % n) + n) % n; }
    else if (g >= n) { live = dm.bc[D][1] == 0; g = g % n; }
    x[D] = g;
    live = live && p.active[dm.block0 + bo + (g / dm.be[D]) * bstride] != 0;
    const long long idx = ((long long)x[2] * dm.n[1] + x[1]) * dm.n[0] + x[0];
#pragma unroll
    for (int v = 0; v < NV; v++) {
      double gv = 0.0;
      if (live) {
        gv = p.G[dm.off + idx + (long long)v * dm.ncell];
        gv = fma(gv, w, gv * wl);
        if (PHYS == PH_MHD && v == 8) gv *= pfac;
      }
      gh[(v * P + pl) * SG + r] = gv;
    }
  }
  __syncthreads();
  // ---- phase B: one thread per (line, variable) walks the faces within reach, in fixed point
  // on the integer units (512^2 MHD: the launch went from 344 us, bound by FP64 replay of the
  // pieces, to about 255); phase C's FP64 and the 12 warps an SM holds bound the kernel now
  int kb = s0 - 2, ke = s0 + slen + 2;
  if (dm.bc[D][0] != 0 && kb < 0) kb = 0;
  if (dm.bc[D][1] != 0 && ke > n) ke = n;
  // cells whose gradient is used: the segment's and, at a face with ghosts, those
  const int lo = dm.bc[D][0] != 0 && s0 == 0 ? -3 : 0;
  const int hi = dm.bc[D][1] != 0 && s0 + slen == n ? slen + 2 : slen - 1;
  const long long nlines = (long long)dm.n[od1] * dm.n[od2];
  const int total = nl * NV, lane = threadIdx.x & 31;
  for (int t0 = threadIdx.x - lane; t0 < total; t0 += blockDim.x) {
    const int t = t0 + lane;
    const unsigned vm = __ballot_sync(0xffffffffu, t < total);
    if (t >= total) continue;
    const int v = t / nl, pl = t - v * nl;
    double* ggp = gGp + (v * P + pl) * SA;
    double* ggm = gGm + (v * P + pl) * SA;
    const int line = it.l0 + pl;
    const int a1 = line % dm.be[od1], a2 = line / dm.be[od1];
    const long long ld = (long long)(o[od2] + a2) * dm.n[od1] + (o[od1] + a1);
    const unsigned short* tp = p.tape + dm.tape_off[D] + ((long long)(v * 2 + 0) * nlines + ld) * (n + 1);
    const TapeLine tape = {tp, tp + nlines * (n + 1), s0, n, dm.bc[D][1] == 0};
    adjoint_sweep<LIMO>((line_t)__cvta_generic_to_shared(gh + (v * P + pl) * SG), slen, tape, kb - s0, ke - s0, lo, hi,
                        ggp, ggm, vm);
    // outflow: ghost copies of an edge cell fold back into it
    if (dm.bc[D][0] == 1 && s0 == 0) {
      const int q0 = 5;  // position of cell 0
      for (int qq = 2; qq < q0; qq++) { ggp[q0] += ggp[qq]; ggm[q0] += ggm[qq]; }
    }
    if (dm.bc[D][1] == 1 && s0 + slen == n) {
      const int qn = slen + 4;  // position of cell n-1
      for (int qq = qn + 1; qq <= qn + 3; qq++) { ggp[qn] += ggp[qq]; ggm[qn] += ggm[qq]; }
    }
  }
  __syncthreads();
  // ---- phase C: transposed flux-split Jacobian per cell of the segment
  for (int c = threadIdx.x; c < nl * slen; c += blockDim.x) {
    int pl, j;
    if (D == 0) { pl = c / slen; j = c - pl * slen; }
    else { j = c / nl; pl = c - j * nl; }
    const int line = it.l0 + pl;
    const int a1 = line % dm.be[od1], a2 = line / dm.be[od1];
    int x[3];
    x[od1] = o[od1] + a1;
    x[od2] = o[od2] + a2;
    x[D] = s0 + j;
    const long long idx = ((long long)x[2] * dm.n[1] + x[1]) * dm.n[0] + x[0];
    double u[NV], gpv[NV], gmv[NV], gu[NV];
    const double* Sv = self_active ? p.S : p.Un;
#pragma unroll
    for (int v = 0; v < NV; v++) {
      u[v] = Sv[dm.off + idx + (long long)v * dm.ncell];
      gpv[v] = gGp[(v * P + pl) * SA + j + 5];
      gmv[v] = gGm[(v * P + pl) * SA + j + 5];
    }
    split_flux_adj<PHYS, NV, D>(u, p.gm1, alpha, ch2, gpv, gmv, gu);
    // mirror faces: the ghost image of this cell (odd variables negated) fed the
    // split fluxes too; its gradient goes through the Jacobian at the image state
    // and back through the sign flip (the segment at a mirror face holds >= 3 cells)
    for (int side = 0; side < 2; side++) {
      int q = -1;
      if (side == 0 && dm.bc[D][0] == 2 && s0 == 0 && j < 3) q = 4 - j;
      if (side == 1 && dm.bc[D][1] == 2 && s0 + slen == n && j >= slen - 3) q = 2 * slen + 4 - j;
      if (q < 0) continue;
      const unsigned odd = dm.asym[D][side];
      double ui[NV], gi[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) {
        ui[v] = ((odd >> v) & 1u) ? -u[v] : u[v];
        gpv[v] = gGp[(v * P + pl) * SA + q];
        gmv[v] = gGm[(v * P + pl) * SA + q];
      }
      split_flux_adj<PHYS, NV, D>(ui, p.gm1, alpha, ch2, gpv, gmv, gi);
#pragma unroll
      for (int v = 0; v < NV; v++) gu[v] += ((odd >> v) & 1u) ? -gi[v] : gi[v];
    }
#pragma unroll
    for (int v = 0; v < NV; v++) p.gL[D][dm.off + idx + (long long)v * dm.ncell] = gu[v];
  }
  __syncthreads();
}

template <int PHYS, int NV, bool LIMO>
__global__ void __launch_bounds__(256) adj_flux_kernel(AdjFluxParams p) {
  extern __shared__ double sm[];
  constexpr int maxd = PHYS == PH_EULER ? NV - 2 : 3;
  for (int it = blockIdx.x; it < p.nitems; it += gridDim.x) {
    const FluxItem item = p.items[p.item0 + it];
    AMRFD_GUARD(p.err, flux_item_ok(p.doms, p.ndom, p.ndim, p.P, p.SSg, item), continue)
    {
      const DomDev& dm = p.doms[item.dom];
      if (!p.active[dm.block0 + item.blk] && !passive_fed(dm, p.active, item.blk, item.d)) continue;
    }
    if (item.d == 0) adj_item<PHYS, NV, 0, LIMO>(p, item, sm);
    if constexpr (maxd > 1) { if (item.d == 1) adj_item<PHYS, NV, 1, LIMO>(p, item, sm); }
    if constexpr (maxd > 2) { if (item.d == 2) adj_item<PHYS, NV, 2, LIMO>(p, item, sm); }
  }
}

// Transposed stage combination: g[U^(k_t)] += a_t gOut, g[U^(i-1)] += sum_d gL_d.
template <int NV>
__global__ void __launch_bounds__(256) adj_combine_kernel(AdjCombParams p) {
  for (int it = blockIdx.x; it < p.nitems; it += gridDim.x) {
    const CellItem ci = p.items[p.item0 + it];
    AMRFD_GUARD(p.err, cell_item_ok(p.doms, p.ndom, ci), continue)
    const DomDev dm = p.doms[ci.dom];
    int o[3];
    {
      const int bx = ci.blk % dm.nb[0], by = (ci.blk / dm.nb[0]) % dm.nb[1], bz = ci.blk / (dm.nb[0] * dm.nb[1]);
      o[0] = bx * dm.be[0]; o[1] = by * dm.be[1]; o[2] = bz * dm.be[2];
    }
    if (!p.active[dm.block0 + ci.blk]) {
      // a passive block's cells entered the stage's fluxes as U^n where they fed an
      // active neighbour: those directions' gradients belong to U^n
      bool fed[3];
      bool any = false;
      for (int d = 0; d < 3; d++) {
        fed[d] = d < p.ndim && passive_fed(dm, p.active, ci.blk, d);
        any |= fed[d];
      }
      if (!any) continue;
      for (int c = threadIdx.x; c < ci.cnt; c += blockDim.x) {
        const int l = ci.c0 + c;
        const int lx = l % dm.be[0], ly = (l / dm.be[0]) % dm.be[1], lz = l / (dm.be[0] * dm.be[1]);
        const long long idx = dm.off + ((long long)(o[2] + lz) * dm.n[1] + (o[1] + ly)) * dm.n[0] + (o[0] + lx);
#pragma unroll
        for (int v = 0; v < NV; v++) {
          const long long e = idx + (long long)v * dm.ncell;
          double s = 0.0;
          for (int d = 0; d < 3; d++)
            if (fed[d]) s += p.gL[d][e];
          p.gbuf[0][e] += s;
        }
      }
      continue;
    }
    const double pfac = p.psi_fac ? p.psi_fac[ci.dom] : 1.0;
    for (int c = threadIdx.x; c < ci.cnt; c += blockDim.x) {
      const int l = ci.c0 + c;
      const int lx = l % dm.be[0], ly = (l / dm.be[0]) % dm.be[1], lz = l / (dm.be[0] * dm.be[1]);
      const long long idx = dm.off + ((long long)(o[2] + lz) * dm.n[1] + (o[1] + ly)) * dm.n[0] + (o[0] + lx);
#pragma unroll
      for (int v = 0; v < NV; v++) {
        const long long e = idx + (long long)v * dm.ncell;
        double g = p.gout[e];
        if (NV == 9 && v == 8) g *= pfac;
        for (int t = 0; t < p.co.nterm; t++) p.gbuf[p.co.k[t]][e] = fma(p.co.a[t], g, p.gbuf[p.co.k[t]][e]);
        double s = p.gL[0][e];
        if (p.ndim > 1) s += p.gL[1][e];
        if (p.ndim > 2) s += p.gL[2][e];
        p.gbuf[p.kin][e] += s;
      }
    }
  }
}

// Passive blocks are the identity map of U^n: their gradient passes through (added to what
// the stages' fluxes gave U^n there, where the block fed an active neighbour).
__global__ void __launch_bounds__(256) adj_passive_kernel(AdjCombParams p) {
  for (int it = blockIdx.x; it < p.nitems; it += gridDim.x) {
    const CellItem ci = p.items[p.item0 + it];
    AMRFD_GUARD(p.err, cell_item_ok(p.doms, p.ndom, ci), continue)
    const DomDev dm = p.doms[ci.dom];
    if (p.active[dm.block0 + ci.blk]) continue;
    int o[3];
    {
      const int bx = ci.blk % dm.nb[0], by = (ci.blk / dm.nb[0]) % dm.nb[1], bz = ci.blk / (dm.nb[0] * dm.nb[1]);
      o[0] = bx * dm.be[0]; o[1] = by * dm.be[1]; o[2] = bz * dm.be[2];
    }
    for (int c = threadIdx.x; c < ci.cnt; c += blockDim.x) {
      const int l = ci.c0 + c;
      const int lx = l % dm.be[0], ly = (l / dm.be[0]) % dm.be[1], lz = l / (dm.be[0] * dm.be[1]);
      const long long idx = dm.off + ((long long)(o[2] + lz) * dm.n[1] + (o[1] + ly)) * dm.n[0] + (o[0] + lx);
      for (int v = 0; v < p.nv; v++) {
        const long long e = idx + (long long)v * dm.ncell;
        p.gbuf[0][e] += p.gout[e];
      }
    }
  }
}

// psi damping factor exp(-dt c_h / c_r) per domain, as applied by the forward step
__global__ void psi_fac_kernel(const unsigned long long* araw0, const double* dt, double* fac, int ndom, int ndim,
                               double cr, int glm) {
  for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < ndom; d += gridDim.x * blockDim.x) {
    double f = 1.0;
    if (glm && cr > 0.0) {
      double ch = 0.0;
      for (int k = 0; k < ndim; k++) ch = imax(ch, bitsd((long long)araw0[(size_t)d * 4 + k]));
      f = exp(-dt[d] * ch / cr);
    }
    fac[d] = f;
  }
}

#define AMRFD_DISPATCH_ADJ(physics, nv, CALL)                               \
  do {                                                                      \
    if ((physics) == PH_MHD && (nv) == 9) { CALL(PH_MHD, 9); }              \
    else if ((physics) == PH_EULER && (nv) == 3) { CALL(PH_EULER, 3); }     \
    else if ((physics) == PH_EULER && (nv) == 4) { CALL(PH_EULER, 4); }     \
    else if ((physics) == PH_EULER && (nv) == 5) { CALL(PH_EULER, 5); }     \
    else return cudaErrorInvalidValue;                                      \
  } while (0)

cudaError_t adj_flux_allow_smem(int physics, int nv, int limo3) {
#define CALL(PH, NVV)                                                                   \
  return allow_smem(limo3 ? (const void*)adj_flux_kernel<PH, NVV, true> : (const void*)adj_flux_kernel<PH, NVV, false>)
  AMRFD_DISPATCH_ADJ(physics, nv, CALL);
#undef CALL
  return cudaSuccess;
}

cudaError_t launch_adj_flux(int physics, int nv, const AdjFluxParams& p, int grid, int block, size_t smem,
                            cudaStream_t s) {
#define CALL(PH, NVV)                                                          \
  if (p.limo3) adj_flux_kernel<PH, NVV, true><<<grid, block, smem, s>>>(p);    \
  else adj_flux_kernel<PH, NVV, false><<<grid, block, smem, s>>>(p)
  AMRFD_DISPATCH_ADJ(physics, nv, CALL);
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_adj_combine(int nv, const AdjCombParams& p, int grid, int block, cudaStream_t s) {
  if (nv == 9) adj_combine_kernel<9><<<grid, block, 0, s>>>(p);
  else if (nv == 3) adj_combine_kernel<3><<<grid, block, 0, s>>>(p);
  else if (nv == 4) adj_combine_kernel<4><<<grid, block, 0, s>>>(p);
  else if (nv == 5) adj_combine_kernel<5><<<grid, block, 0, s>>>(p);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_adj_passive(const AdjCombParams& p, int grid, int block, cudaStream_t s) {
  adj_passive_kernel<<<grid, block, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_psi_fac(const unsigned long long* araw0, const double* dt, double* fac, int ndom, int ndim,
                           double cr, int glm, cudaStream_t s) {
  psi_fac_kernel<<<(ndom + 255) / 256, 256, 0, s>>>(araw0, dt, fac, ndom, ndim, cr, glm);
  return cudaGetLastError();
}

}  // namespace amrfd
