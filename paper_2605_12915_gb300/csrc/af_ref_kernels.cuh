// af_ref_kernels.cuh -- the RB-TAI / RB step as separate kernels, one thread per
// node or cell, intermediate values in global scratch.  It is the FP64 path and
// the reference layout for the fused kernel:
//   k_center    centre recovery by Simpson inversion        (Eq. center-node)
//   k_acoustic  node-centred exact acoustic increments      (Sec. 6.1 step 1)
//   k_points    two-Picard foot + transported / additive    (Sec. 6.1 steps 2-4,
//               point update at tau = dt/2 and dt           Eq. barsukow-additive)
//               and the time-integrated fluxes of the node  (Sec. 3.1)
//   k_average   conservative average update                 (Eq. af-average-update)
//
// What bounds them in FP64: the FP64 unit, two lanes per cycle and SM, so a warp
// instruction holds its scheduler's unit for 64 cycles while everything else
// (loads, integer work, launches of other warps) is all but free.  Comparisons,
// conversions, floor and min / max of doubles run on that unit too.  So the FP64
// instructions are what is counted here: comparisons and floor are done on the
// bits, increments are kept as
// (u + du, v + dv, dp) and interpolated together with the velocity (five fields
// at the foot instead of seven), and each
// node's fluxes are integrated in time once instead of in both edges it bounds.
// Small grids are bound by the same unit on the few SMs that hold their warps:
// the families share a launch (blockIdx.y) and blocks are two warps.
// GB300, FP64: a step at 512^2 takes 1.07 ms (1.40 with ten launches, comparisons
// and floor in FP64, separate increments and per-edge fluxes); a whole
// set-step-get call at 32^2 from pinned host memory 76 us (277).  (Shorter forms of the
// centre recovery, the freezing and the interpolation at the foot made it 1.01 ms and 71
// us, but rounded more; see there.)
#pragma once

#include "af_common.cuh"
#include "af_stencils.cuh"

namespace af {

template <typename T>
struct StepArgs {
  Planes<T> in;       // state at t^n
  Planes<T> out;      // state at t^{n+1}
  T* wc[4];           // recovered centre (rho, u, v, p)
  T* inc[2][4][3];    // [tau index][family V,Ev,Eh,C][u + du, v + dv, dp] (RB: du, dv, dp)
  T* half[3][4];      // point values at t^n + dt/2, [family][rho,u,v,p] (adjoint and AF_FC);
                      // the step keeps the fluxes of the vertices (x, then y) and of the
                      // x-edge midpoints there
  T* fx[4];           // fluxes of the y-edge midpoints
  unsigned* flags;
  int nx, ny;
  T h, dt, dth;       // dth = dt / h
  Gas<T> gas;
  int variant;        // 0 TAI, 1 RB
  int prefetch_wave;  // fused kernel: blocks per wave for the L2 prefetch (0: none)
  int late_first_wait;  // pipelined kernels, testing only: each CTA's first wait for a
                        // tensor-copied tile reports a timeout at once (0: off)
};

constexpr int REF_THREADS = 64;

template <typename T>
__device__ __forceinline__ LatticeG<T> lattice_of(const StepArgs<T>& a) {
  LatticeG<T> L;
  for (int f = 0; f < 3; ++f)
    for (int k = 0; k < 4; ++k) L.f[f][k] = a.in.pt[f][k];
  for (int k = 0; k < 4; ++k) L.f[3][k] = a.wc[k];
  L.nx = a.nx;
  L.ny = a.ny;
  return L;
}

__device__ __forceinline__ void raise_flag(unsigned* flags, unsigned bits) {
  if (bits) atomicOr(flags, bits);
}

// family of lattice offset (a, b) from a cell's vertex: V, E_v, E_h, C
__host__ __device__ constexpr int fam_of(int a, int b) {
  return (a & 1) ? ((b & 1) ? 3 : 2) : ((b & 1) ? 1 : 0);
}

// the calling thread's cell (false: beyond the grid)
template <typename T>
__device__ __forceinline__ bool cell_of_thread(const StepArgs<T>& a, int& i, int& j, size_t& id) {
  id = (size_t)blockIdx.x * REF_THREADS + threadIdx.x;
  if (id >= (size_t)a.nx * a.ny) return false;
  j = (int)(id / (unsigned)a.nx);
  i = (int)(id - (size_t)j * a.nx);
  return true;
}

// Wrapped neighbourhood of cell (ci, cj): columns ci-1, ci, ci+1 and row
// offsets (cj-1) nx, cj nx, (cj+1) nx; a lattice offset resolves at compile
// time to one of them.
struct Nbhd {
  int col[3];
  size_t row[3];
  __device__ __forceinline__ size_t at(int dc, int dr) const { return row[dr + 1] + col[dc + 1]; }
};

__device__ __forceinline__ Nbhd nbhd(int ci, int cj, int nx, int ny) {
  Nbhd b;
  b.col[1] = ci;
  b.col[0] = ci == 0 ? nx - 1 : ci - 1;
  b.col[2] = ci + 1 == nx ? 0 : ci + 1;
  const int rm = cj == 0 ? ny - 1 : cj - 1, rp = cj + 1 == ny ? 0 : cj + 1;
  b.row[0] = (size_t)rm * nx;
  b.row[1] = (size_t)cj * nx;
  b.row[2] = (size_t)rp * nx;
  return b;
}

// ---------------------------------------------------------------------------
// Centre recovery (Eq. center-node) in the deviation form
// U_c = Ubar + 1/16 sum_corners (Ubar - U_V) + 1/4 sum_edges (Ubar - U_E): its
// roundings are those of the deviations, where U_c = 9/4 Ubar - sum_corners U_V / 16 -
// sum_edges U_E / 4 (36 FP64 instructions instead of 68) rounds sums four times
// as large as U and has twice the error.
// ---------------------------------------------------------------------------
// TOP: also raises *top.bits to the bits of the largest FP32 wave speed of the cell's
// own nodes (positive floats compare as their bits).
struct TopSpeed {
  unsigned* bits;
  RefPair rho_ref, p_ref;
  float gamma;
};
template <typename T, bool COMP, bool TOP = false>
__global__ void __launch_bounds__(REF_THREADS)
    k_center(const __grid_constant__ StepArgs<T> a, const __grid_constant__ TopSpeed top) {
  pdl_wait();
  int i, j;
  size_t id;
  if (!cell_of_thread(a, i, j, id)) return;
  const int ip = i + 1 == a.nx ? 0 : i + 1, jp = j + 1 == a.ny ? 0 : j + 1;
  auto P = [&](int f, int ii, int jj) {
    size_t q = (size_t)jj * a.nx + ii;
    Prim<T> w = {a.in.pt[f][0][q], a.in.pt[f][1][q], a.in.pt[f][2][q], a.in.pt[f][3][q]};
    return w;
  };
  T ub[4], lo[4], uc[4], c[4], e[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    ub[k] = a.in.avg[k][id];
    lo[k] = COMP ? a.in.lo[k][id] : T(0);
  }
  // the sum of the first n deviations and the next one
  auto dev = [](T ubar, T u, T l, int n, T sum) {
    const T d = COMP ? (ubar - u) + l : ubar - u;
    return n == 0 ? d : sum + d;
  };
  const Prim<T> corners[4] = {P(0, i, j), P(0, ip, j), P(0, i, jp), P(0, ip, jp)};
  const Prim<T> edges[4] = {P(2, i, j), P(2, i, jp), P(1, i, j), P(1, ip, j)};
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    T u[4];
    cons_from_stored(corners[n], a.gas, u);
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = dev(ub[k], u[k], lo[k], n, c[k]);
    cons_from_stored(edges[n], a.gas, u);
#pragma unroll
    for (int k = 0; k < 4; ++k) e[k] = dev(ub[k], u[k], lo[k], n, e[k]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    uc[k] = (COMP ? ub[k] + lo[k] : ub[k]) + fma(T(0.0625), c[k], T(0.25) * e[k]);
  Prim<T> w = stored_from_cons(uc, a.gas);
  a.wc[0][id] = w.r;
  a.wc[1][id] = w.u;
  a.wc[2][id] = w.v;
  a.wc[3][id] = w.p;
  if constexpr (TOP) {
    auto speed = [&](const Prim<T>& n) {
      const float s = wave_speed_f32(top.rho_ref, top.p_ref, n.r, n.u, n.v, n.p, top.gamma);
      return s < INFINITY ? s : 0.f;  // (the reduction looks at the others itself)
    };
    const float s = fmaxf(fmaxf(speed(corners[0]), speed(edges[0])),
                          fmaxf(speed(edges[2]), speed(w)));
    const unsigned m = __reduce_max_sync(__activemask(), __float_as_uint(s));
    if (m > *(volatile unsigned*)top.bits) atomicMax(top.bits, m);
  }
  raise_flag(a.flags, (is_positive(with_ref(a.gas.rho_ref, w.r)) &&
                       is_positive(with_ref(a.gas.p_ref, w.p)))
                          ? 0u
                          : FLAG_NONPHYSICAL);
}

// ---------------------------------------------------------------------------
// Exact frozen acoustic increments of the nodes of the family blockIdx.y, for
// tau = dt/2 and tau = dt (Sec. 6.1 step 1).  The r^q sums are shared by both.
// ---------------------------------------------------------------------------
// node values (.p, .u, .v) at lattice offset (dx, dy) from the node of family
// FAM of the neighbourhood's centre cell
template <int FAM, typename T>
struct LoadPUV {
  const StepArgs<T>* a;
  Nbhd b;
  __device__ __forceinline__ PUV<T> operator()(int dx, int dy) const {
    const int ax = ((FAM == 2 || FAM == 3) ? 1 : 0) + dx, by = ((FAM == 1 || FAM == 3) ? 1 : 0) + dy;
    const int f = fam_of(ax, by);
    const size_t q = b.at(ax >> 1, by >> 1);
    T* const* pl = f < 3 ? a->in.pt[f] : a->wc;
    PUV<T> o = {pl[3][q], pl[1][q], pl[2][q]};
    return o;
  }
};

template <int FAM, typename T, typename Load>
__device__ __forceinline__ void sac_family(const Load& L, T pK, T uK, T vK, T Gp[3][4],
                                           T Guv[3][4]) {
  if constexpr (FAM == 0) af_sac_V<T>(L, pK, uK, vK, Gp, Guv);
  if constexpr (FAM == 1) af_sac_EV<T>(L, pK, uK, vK, Gp, Guv);
  if constexpr (FAM == 2) af_sac_EH<T>(L, pK, uK, vK, Gp, Guv);
  if constexpr (FAM == 3) af_sac_C<T>(L, pK, uK, vK, Gp, Guv);
}

// The frozen sound speed c = sqrt(gamma p / rho), impedance Z = rho c and 1 / Z of a
// node, each rounded by IEEE operations.  (One reciprocal root, 1/Z =
// rsqrt(gamma p rho), saves the root and two divisions but doubles the error of c and
// leaves the exponent range where p rho does.)
template <typename T>
__device__ __forceinline__ void freeze(T gamma, T rho, T p, T& c, T& Z, T& Zinv) {
  c = sqrt(gamma * p / rho);
  Z = rho * c;
  Zinv = T(1) / Z;
}

template <int FAM, typename T>
__device__ __forceinline__ void acoustic_node(const StepArgs<T>& a, int i, int j, size_t id) {
  T* const* own = FAM < 3 ? a.in.pt[FAM < 3 ? FAM : 0] : a.wc;
  const Prim<T> wk = {own[0][id], own[1][id], own[2][id], own[3][id]};
  unsigned bad = 0;
  const T rk = with_ref(a.gas.rho_ref, wk.r), pk = with_ref(a.gas.p_ref, wk.p);
  if (!(is_positive(rk) && is_positive(pk))) bad |= FLAG_NONPHYSICAL;
  T c, Z, Zinv;
  freeze(a.gas.gamma, rk, pk, c, Z, Zinv);
  const T r1 = c * a.dth;
  if (abs_above(r1, T(0.5))) bad |= FLAG_CFL;
  T Gp[3][4], Guv[3][4];
  const LoadPUV<FAM, T> ld = {&a, nbhd(i, j, a.nx, a.ny)};
  sac_family<FAM, T>(ld, wk.p, wk.u, wk.v, Gp, Guv);
  // polynomial coefficients: dp = sum_q r^q (Gp0 + Z Guv0), du = sum_q r^q (Gp1 / Z + Guv1)
  T cp[4], cu[4], cv[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    cp[q] = fma(Z, Guv[0][q], Gp[0][q]);
    cu[q] = fma(Zinv, Gp[1][q], Guv[1][q]);
    cv[q] = fma(Zinv, Gp[2][q], Guv[2][q]);
  }
  // (the additive update takes the increments at the point itself, without interpolation:
  // kept alone there, they do not carry a rounding of the velocity)
  const T u0 = a.variant == 0 ? wk.u : T(0), v0 = a.variant == 0 ? wk.v : T(0);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const T r = s == 0 ? T(0.5) * r1 : r1;
    a.inc[s][FAM][0][id] = fma(r, fma(r, fma(r, fma(r, cu[3], cu[2]), cu[1]), cu[0]), u0);
    a.inc[s][FAM][1][id] = fma(r, fma(r, fma(r, fma(r, cv[3], cv[2]), cv[1]), cv[0]), v0);
    a.inc[s][FAM][2][id] = r * fma(r, fma(r, fma(r, cp[3], cp[2]), cp[1]), cp[0]);
  }
  raise_flag(a.flags, bad);
}

template <typename T>
__global__ void __launch_bounds__(REF_THREADS) k_acoustic(const __grid_constant__ StepArgs<T> a) {
  pdl_wait();
  int i, j;
  size_t id;
  if (!cell_of_thread(a, i, j, id)) return;
  switch (blockIdx.y) {
    case 0: acoustic_node<0>(a, i, j, id); break;
    case 1: acoustic_node<1>(a, i, j, id); break;
    case 2: acoustic_node<2>(a, i, j, id); break;
    default: acoustic_node<3>(a, i, j, id); break;
  }
}

// ---------------------------------------------------------------------------
// Point update (Sec. 6.1 steps 3-4).  Positions are kept as an integer cell
// index plus a small offset so that FP32 resolves the foot on large grids.
// ---------------------------------------------------------------------------
template <typename T>
struct FootCell {
  int ci, cj;  // cell containing the point
  T xi, eta;   // local coordinates in [-1, 1]
};

// point at lattice (I, J) displaced by (dx, dy) cells
template <typename T>
__device__ __forceinline__ FootCell<T> locate(int I, int J, T dx, T dy) {
  T fx = T(0.5) * (T)(I & 1) + dx;
  T fy = T(0.5) * (T)(J & 1) + dy;
  T flx = floor(fx), fly = floor(fy);
  FootCell<T> c;
  c.ci = (I >> 1) + (int)flx;
  c.cj = (J >> 1) + (int)fly;
  c.xi = T(2) * (fx - flx) - T(1);
  c.eta = T(2) * (fy - fly) - T(1);
  return c;
}

template <typename T>
__device__ __forceinline__ Prim<T> eval_w(const LatticeG<T>& L, const FootCell<T>& c) {
  T lx[3], ly[3];
  lagrange3(c.xi, lx);
  lagrange3(c.eta, ly);
  Prim<T> s = {T(0), T(0), T(0), T(0)};
  for (int b = 0; b < 3; ++b) {
    Prim<T> row = {T(0), T(0), T(0), T(0)};
    for (int q = 0; q < 3; ++q) {
      Prim<T> w = L.at(2 * c.ci + q, 2 * c.cj + b);
      row.r = fma(lx[q], w.r, row.r);
      row.u = fma(lx[q], w.u, row.u);
      row.v = fma(lx[q], w.v, row.v);
      row.p = fma(lx[q], w.p, row.p);
    }
    s.r = fma(ly[b], row.r, s.r);
    s.u = fma(ly[b], row.u, s.u);
    s.v = fma(ly[b], row.v, s.v);
    s.p = fma(ly[b], row.p, s.p);
  }
  return s;
}

// One axis of a foot displaced by d cells from lattice offset O (0 or 1 half
// cell): the cell offset floor(f), f = O/2 + d, and the local coordinate
// 2 (f - floor(f)) - 1.  Within the reach (|d| <= 1) floor(f) is -1, 0 or 1,
// read off the bits; beyond it (flagged by the caller) by floor itself.
template <int O, typename T>
__device__ __forceinline__ T foot_coord(T d, int& cell) {
  const T f = O ? d + T(0.5) : d;
  if (abs_above(d, T(1)) || !is_finite(d)) {
    const T fl = floor(f);
    cell = (int)fl;
    return fma(T(2), f - fl, T(-1));
  }
  const bool neg = is_negative(f), one = at_least_one(f);
  cell = neg ? -1 : (one ? 1 : 0);
  return fma(T(2), f, neg ? T(1) : (one ? T(-3) : T(-1)));
}

template <typename T>
__device__ __forceinline__ void lagrange3_fma(T s, T l[3]) {
  const T hs = T(0.5) * s;
  l[0] = fma(hs, s, -hs);
  l[1] = fma(-s, s, T(1));
  l[2] = fma(hs, s, hs);
}

// the cells (c0, c0 + 1) x (r0, r0 + 1), wrapped, that hold the nine nodes of the
// cell (i + cx, j + cy): node (q, b) is the family fam_of(q, b) of cell n[b / 2][q / 2]
struct FootNodes {
  size_t n[2][2];
};
__device__ __forceinline__ FootNodes foot_nodes(int c, int r, int nx, int ny) {
  if ((unsigned)(c + 1) > (unsigned)nx) c = wrapi(c, nx);  // beyond [-1, nx)
  if ((unsigned)(r + 1) > (unsigned)ny) r = wrapi(r, ny);
  c = c < 0 ? c + nx : (c == nx ? 0 : c);
  r = r < 0 ? r + ny : (r == ny ? 0 : r);
  const size_t r0 = (size_t)r * nx, r1 = r + 1 == ny ? 0 : r0 + nx;
  const int c1 = c + 1 == nx ? 0 : c + 1;
  FootNodes f = {{{r0 + c, r0 + c1}, {r1 + c, r1 + c1}}};
  return f;
}

// sum_qb lx_q ly_b f_qb with f_qb the plane of the node's family, pl(fam): rows first.
// (Nine products with the weights lx_q ly_b formed once for all fields take 9 FP64
// instructions instead of 12, but round each weight and eight sums of full size: 5 to
// 14% more error in the density and pressure at the foot.)
template <typename T, typename Plane>
__device__ __forceinline__ T row_sum(const FootNodes& c, const T lx[3], const T ly[3],
                                     const Plane& pl) {
  T r[3];
#pragma unroll
  for (int b = 0; b < 3; ++b)
    r[b] = fma(lx[2], pl(fam_of(2, b))[c.n[b >> 1][1]],
               fma(lx[1], pl(fam_of(1, b))[c.n[b >> 1][0]],
                   lx[0] * pl(fam_of(0, b))[c.n[b >> 1][0]]));
  return fma(ly[2], r[2], fma(ly[1], r[1], ly[0] * r[0]));
}

// Adds wt times the node's fluxes (x for V and E_v, y for V and E_h) to S.
template <int FAM, typename T>
__device__ __forceinline__ void add_flux(const Prim<T>& w, const Gas<T>& g, T wt, T S[2][4]) {
  T f[4];
  if (FAM != 2) {
    flux_x(w, g, f);
#pragma unroll
    for (int k = 0; k < 4; ++k) S[0][k] = fma(wt, f[k], S[0][k]);
  }
  if (FAM != 1) {
    flux_y(w, g, f);
#pragma unroll
    for (int k = 0; k < 4; ++k) S[1][k] = fma(wt, f[k], S[1][k]);
  }
}

// Point of family FAM of cell (i, j), both durations.  FLUX: the half-step point
// stays in registers and the node's fluxes, summed over time with weights
// 1, 4, 1, are stored; otherwise the half-step point is (for the adjoint).
template <int FAM, bool FLUX, typename T>
__device__ __forceinline__ void point_node(const StepArgs<T>& a, int i, int j, size_t id) {
  const int nx = a.nx, ny = a.ny;
  const Gas<T>& g = a.gas;
  constexpr int OX = FAM == 2 ? 1 : 0, OY = FAM == 1 ? 1 : 0;
  const Prim<T> wp = {a.in.pt[FAM][0][id], a.in.pt[FAM][1][id], a.in.pt[FAM][2][id],
                      a.in.pt[FAM][3][id]};
  unsigned bad = 0;
  T S[2][4] = {};
  if (FLUX) add_flux<FAM>(wp, g, T(1), S);
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const T th = s == 0 ? T(0.5) * a.dth : a.dth;
    auto plane = [&](int k) {
      return [&a, k](int f) { return f < 3 ? a.in.pt[f][k] : a.wc[k]; };
    };
    auto incr = [&](int k) { return [&a, s, k](int f) { return a.inc[s][f][k]; }; };
    // two-Picard convective foot from the time-n reconstruction (Eq. adv-footpoint)
    int cx, cy;
    T lx[3], ly[3];
    const T d1x = -th * wp.u, d1y = -th * wp.v;
    lagrange3_fma(foot_coord<OX>(d1x, cx), lx);
    lagrange3_fma(foot_coord<OY>(d1y, cy), ly);
    FootNodes c = foot_nodes(i + cx, j + cy, nx, ny);
    const T dfx = -th * row_sum(c, lx, ly, plane(1)), dfy = -th * row_sum(c, lx, ly, plane(2));
    if (abs_above(d1x, T(1)) || abs_above(d1y, T(1)) || abs_above(dfx, T(1)) ||
        abs_above(dfy, T(1)))
      bad |= FLAG_REACH;
    lagrange3_fma(foot_coord<OX>(dfx, cx), lx);
    lagrange3_fma(foot_coord<OY>(dfy, cy), ly);
    c = foot_nodes(i + cx, j + cy, nx, ny);
    const T rft = row_sum(c, lx, ly, plane(0)), pft = row_sum(c, lx, ly, plane(3));
    Prim<T> nw;
    if (a.variant == 0) {
      // transported increment evaluated at the foot; rho from dp / c_f^2.  The
      // velocity's increments are interpolated together with it: u_f + du_f =
      // I_h(u + du)(P_f), both interpolants sharing the basis
      const T dp = row_sum(c, lx, ly, incr(2));
      const T rf = with_ref(g.rho_ref, rft), pf = with_ref(g.p_ref, pft);
      if (!(is_positive(rf) && is_positive(pf))) bad |= FLAG_NONPHYSICAL;
      nw.r = rft + dp * rf / (g.gamma * pf);
      nw.u = row_sum(c, lx, ly, incr(0));
      nw.v = row_sum(c, lx, ly, incr(1));
      nw.p = pft + dp;
    } else {
      // additive update: S_ac(P) + S_adv(P) - W(P), acoustic rho closure at P
      const T dp = a.inc[s][FAM][2][id];
      nw.r = rft + dp * with_ref(g.rho_ref, wp.r) / (g.gamma * with_ref(g.p_ref, wp.p));
      nw.u = row_sum(c, lx, ly, plane(1)) + a.inc[s][FAM][0][id];
      nw.v = row_sum(c, lx, ly, plane(2)) + a.inc[s][FAM][1][id];
      nw.p = pft + dp;
    }
    if (!(is_finite(nw.r) && is_finite(nw.u) && is_finite(nw.v) && is_finite(nw.p)))
      bad |= FLAG_NONFINITE;
    if (FLUX) add_flux<FAM>(nw, g, s == 0 ? T(4) : T(1), S);
    if (s == 1 || !FLUX) {
      T* const* dst = s == 0 ? a.half[FAM] : a.out.pt[FAM];
      dst[0][id] = nw.r;
      dst[1][id] = nw.u;
      dst[2][id] = nw.v;
      dst[3][id] = nw.p;
    }
  }
  if (FLUX) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (FAM == 0) {
        a.half[0][k][id] = S[0][k];
        a.half[1][k][id] = S[1][k];
      } else if (FAM == 1) {
        a.half[2][k][id] = S[0][k];
      } else {
        a.fx[k][id] = S[1][k];
      }
    }
  }
  raise_flag(a.flags, bad);
}

template <typename T, bool FLUX>
__global__ void __launch_bounds__(REF_THREADS) k_points(const __grid_constant__ StepArgs<T> a) {
  pdl_wait();
  int i, j;
  size_t id;
  if (!cell_of_thread(a, i, j, id)) return;
  switch (blockIdx.y) {
    case 0: point_node<0, FLUX>(a, i, j, id); break;
    case 1: point_node<1, FLUX>(a, i, j, id); break;
    default: point_node<2, FLUX>(a, i, j, id); break;
  }
}

// ---------------------------------------------------------------------------
// Time-integrated fluxes of the nodes (weights 1, 4, 1) and the average update.
// ---------------------------------------------------------------------------
template <typename T>
struct NodeFlux {
  T *vx[4], *vy[4], *ex[4], *ey[4];  // V (x, y), E_v (x), E_h (y), per component
};

// the planes k_points<T, true> stores them in
template <typename T>
inline NodeFlux<T> node_flux_of(const StepArgs<T>& a) {
  NodeFlux<T> n;
  for (int k = 0; k < 4; ++k) {
    n.vx[k] = a.half[0][k];
    n.vy[k] = a.half[1][k];
    n.ex[k] = a.half[2][k];
    n.ey[k] = a.fx[k];
  }
  return n;
}

// ... of states whose half-step points are in a.half (AF_FC)
template <typename T>
__global__ void __launch_bounds__(REF_THREADS)
    k_node_flux(const __grid_constant__ StepArgs<T> a, const __grid_constant__ NodeFlux<T> n) {
  pdl_wait();
  int i, j;
  size_t id;
  if (!cell_of_thread(a, i, j, id)) return;
  auto node = [&](T* const* pl) {
    Prim<T> w = {pl[0][id], pl[1][id], pl[2][id], pl[3][id]};
    return w;
  };
  T SV[2][4] = {}, SX[2][4] = {}, SY[2][4] = {};
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    T* const* const lev[3] = {s == 0 ? a.in.pt[0] : s == 1 ? a.half[0] : a.out.pt[0],
                              s == 0 ? a.in.pt[1] : s == 1 ? a.half[1] : a.out.pt[1],
                              s == 0 ? a.in.pt[2] : s == 1 ? a.half[2] : a.out.pt[2]};
    const T wt = s == 1 ? T(4) : T(1);
    add_flux<0>(node(lev[0]), a.gas, wt, SV);
    add_flux<1>(node(lev[1]), a.gas, wt, SX);
    add_flux<2>(node(lev[2]), a.gas, wt, SY);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    n.vx[k][id] = SV[0][k];
    n.vy[k][id] = SV[1][k];
    n.ex[k][id] = SX[0][k];
    n.ey[k][id] = SY[1][k];
  }
}

// Conservative average update (Eq. af-average-update): the edges' Simpson sums of
// their nodes' fluxes, each formed the same way in the two cells it bounds.
// COMP: hi + lo pairs updated by error-free sums of the four edge terms, so that
// each edge value enters its two cells with opposite signs exactly.
template <typename T, bool COMP>
__global__ void __launch_bounds__(REF_THREADS)
    k_average(const __grid_constant__ StepArgs<T> a, const __grid_constant__ NodeFlux<T> n) {
  pdl_wait();
  int i, j;
  size_t id;
  if (!cell_of_thread(a, i, j, id)) return;
  const int ip = i + 1 == a.nx ? 0 : i + 1, jp = j + 1 == a.ny ? 0 : j + 1;
  const size_t up = (size_t)jp * a.nx + i, rt = (size_t)j * a.nx + ip, ur = (size_t)jp * a.nx + ip;
  const T lam = a.dth / T(36);
  unsigned bad = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const T *vx = n.vx[k], *vy = n.vy[k], *ex = n.ex[k], *ey = n.ey[k];
    // edge sums at x_i, x_{i+1}, y_j, y_{j+1}
    T fl = fma(T(4), ex[id], vx[id] + vx[up]), fr = fma(T(4), ex[rt], vx[rt] + vx[ur]);
    T gb = fma(T(4), ey[id], vy[id] + vy[rt]), gt = fma(T(4), ey[up], vy[up] + vy[ur]);
    if constexpr (COMP) {
      float hi = a.in.avg[k][id], lo = a.in.lo[k][id];
      comp_update(hi, lo, lam * fl, lam * fr, lam * gb, lam * gt);
      a.out.avg[k][id] = hi;
      a.out.lo[k][id] = lo;
      if (!is_finite(hi)) bad |= FLAG_NONFINITE;
    } else {
      const T v = fma(-lam, (fr - fl) + (gt - gb), a.in.avg[k][id]);
      a.out.avg[k][id] = v;
      if (!is_finite(v)) bad |= FLAG_NONFINITE;
    }
  }
  raise_flag(a.flags, bad);
}

}  // namespace af
