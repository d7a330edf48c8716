// af_adjoint.cuh -- hand-written discrete adjoint of one step (Sec. 6.1):
// lambda^n = (d state^{n+1} / d state^n)^T lambda^{n+1}, linearised about the
// state at t^n.  The forward intermediates are recomputed (the fused kernel's
// tiles, or the kernels of af_ref_kernels.cuh); the reverse sweep then runs
//   points      the space-time Simpson fluxes the point enters (a gather from the
//               averages' lambda) and its transported / additive update: the Q2
//               evaluation at the foot and the two Picard stages, both durations
//               (k_adj_points, or tile_reverse in the fused sweeps)
//   k_adj_acoustic  Horner in r, node freezing (c, Z, r) and the transposed
//                   acoustic stencils (all four node families)
//   k_adj_center, k_adj_out  Simpson inversion, lambda^n out
// The scatters add each contribution to global memory with one vector reduction:
// the adjoints of the lattice nodes and of the increments are kept as 4-wide
// records per node (FP32: one float4 atomic), which start at zero and are cleared
// by the kernel that consumes them.  Adjoints are with respect to the stored
// variables; the storage offsets of the FP32 modes are constant shifts and do not
// change them.
#pragma once

#include "af_common.cuh"
#include "af_fused.cuh"
#include "af_launch.cuh"
#include "af_ref_kernels.cuh"

namespace af {

// Planes of one adjoint step, all with one stride (elements) from three bases.
template <typename T>
struct AdjView {
  const T* st;   // state^n: averages 0-3, points 4 + 4 fam + k
  const T* sto;  // state^{n+1} of the recomputed step: same layout
  const T* scr;  // intermediates: centres 0-3, increments 4 + 12 s + 3 fam + k,
                 // half-step points 28 + 4 fam + k
  T* lam;        // adjoints, in units of ps: lambda^n of the averages 0-3 (planes);
                 // node records of family fam at 4 + 4 fam (4 values per cell: rho,
                 // u, v, p; family 3 is the centre); increment records of (s, fam)
                 // at 20 + 4 (4 s + fam) (du, dv, dp, 0); the centre adjoint
                 // lambda_U of each cell 52 + k (planes)
  size_t ps;
  int nx, ny;
  T h, dt, dth;  // dth = dt / h
  Gas<T> gas;
  int variant;
  const double* lin64[16];  // lambda^{n+1} as given (FP64 device planes)
};

constexpr int LAM_OUT = 0, LAM_NODE = 4, LAM_INC = 20, LAM_LU = 52;
constexpr int LAM_PLANES = 56;
constexpr int SCR_INC = 4, SCR_HALF = 28;

// cell index wrapped into [0, n): one conditional step for |i| < 2n
__device__ __forceinline__ int wrapc(int i, int n) {
  const int w = i < 0 ? i + n : (i >= n ? i - n : i);
  return (unsigned)w < (unsigned)n ? w : wrapi(i, n);
}

template <typename T>
__device__ __forceinline__ size_t cell_id(const AdjView<T>& v, int cx, int cy) {
  return (size_t)wrapc(cy, v.ny) * v.nx + wrapc(cx, v.nx);
}

// time-n value (rho~, u, v, p~) of the node of family fam of cell id
template <typename T>
__device__ __forceinline__ Prim<T> node_w(const AdjView<T>& v, int fam, size_t id) {
  const T* b = fam < 3 ? v.st + (size_t)(4 + 4 * fam) * v.ps : v.scr;
  Prim<T> w = {b[id], b[v.ps + id], b[2 * v.ps + id], b[3 * v.ps + id]};
  return w;
}

// adds (a, b, c, d) to the 4-wide record at p (16-byte aligned), without
// looking for zeros
__device__ __forceinline__ void add4_always(float* p, float a, float b, float c, float d) {
  atomicAdd(reinterpret_cast<float4*>(p), make_float4(a, b, c, d));
}
__device__ __forceinline__ void add4_always(double* p, double a, double b, double c, double d) {
  atomicAdd(p, a);
  atomicAdd(p + 1, b);
  atomicAdd(p + 2, c);
  atomicAdd(p + 3, d);
}

// the same for the three values of an increment record
__device__ __forceinline__ void add3_always(float* p, float a, float b, float c) {
  atomicAdd(reinterpret_cast<float4*>(p), make_float4(a, b, c, 0.f));
}
__device__ __forceinline__ void add3_always(double* p, double a, double b, double c) {
  atomicAdd(p, a);
  atomicAdd(p + 1, b);
  atomicAdd(p + 2, c);
}

// clears the 4-wide record at p once its consumer has read it, so that the
// records start the next adjoint step at zero without a separate clearing pass
__device__ __forceinline__ void zero4(float* p) {
  *reinterpret_cast<float4*>(p) = make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void zero4(double* p) {
  reinterpret_cast<double2*>(p)[0] = make_double2(0.0, 0.0);
  reinterpret_cast<double2*>(p)[1] = make_double2(0.0, 0.0);
}

// adds (a, b, c, d) to the 4-wide record at p (16-byte aligned)
__device__ __forceinline__ void add4(float* p, float a, float b, float c, float d) {
  if (a != 0.f || b != 0.f || c != 0.f || d != 0.f)
    atomicAdd(reinterpret_cast<float4*>(p), make_float4(a, b, c, d));
}
__device__ __forceinline__ void add4(double* p, double a, double b, double c, double d) {
  if (a != 0.0) atomicAdd(p, a);
  if (b != 0.0) atomicAdd(p + 1, b);
  if (c != 0.0) atomicAdd(p + 2, c);
  if (d != 0.0) atomicAdd(p + 3, d);
}

// Transposed Euler flux Jacobians: o += J_F(w)^T l  (stored primitives)
template <typename T>
__device__ __forceinline__ void flux_x_adj(const Prim<T>& w, const Gas<T>& g, const T l[4],
                                           T o[4]) {
  const T rho = with_ref(g.rho_ref, w.r), p = with_ref(g.p_ref, w.p);
  const T ke = T(0.5) * fma(w.u, w.u, w.v * w.v), hh = fma(p, g.g_gm1, rho * ke);
  const T t = fma(w.v, l[2], fma(w.u, l[1], l[0]));
  o[0] = fma(w.u, fma(ke, l[3], t), o[0]);
  o[1] = fma(rho, fma(w.u, fma(w.u, l[3], l[1]), t), fma(hh, l[3], o[1]));
  o[2] = fma(rho * w.u, fma(w.v, l[3], l[2]), o[2]);
  o[3] = fma(g.g_gm1 * w.u, l[3], o[3] + l[1]);
}

template <typename T>
__device__ __forceinline__ void flux_y_adj(const Prim<T>& w, const Gas<T>& g, const T l[4],
                                           T o[4]) {
  const T rho = with_ref(g.rho_ref, w.r), p = with_ref(g.p_ref, w.p);
  const T ke = T(0.5) * fma(w.u, w.u, w.v * w.v), hh = fma(p, g.g_gm1, rho * ke);
  const T t = fma(w.v, l[2], fma(w.u, l[1], l[0]));
  o[0] = fma(w.v, fma(ke, l[3], t), o[0]);
  o[1] = fma(rho * w.v, fma(w.u, l[3], l[1]), o[1]);
  o[2] = fma(rho, fma(w.v, fma(w.v, l[3], l[2]), t), fma(hh, l[3], o[2]));
  o[3] = fma(g.g_gm1 * w.v, l[3], o[3] + l[2]);
}

// derivative of the Lagrange basis l_-, l_0, l_+ with respect to s
template <typename T>
__device__ __forceinline__ void lagrange3_d(T s, T d[3]) {
  d[0] = s - T(0.5);
  d[1] = T(-2) * s;
  d[2] = s + T(0.5);
}

template <typename T>
__device__ __forceinline__ void dcons_dprim_T(const Prim<T>& w, const Gas<T>& g, const T l[4],
                                              T s, T o[4]) {
  // o += s (dU/dW)^T l, U = (rho~, rho u, rho v, E~) of the stored primitive
  const T rho = s * with_ref(g.rho_ref, w.r), ke = T(0.5) * fma(w.u, w.u, w.v * w.v);
  o[0] = fma(s, fma(ke, l[3], fma(w.v, l[2], fma(w.u, l[1], l[0]))), o[0]);
  o[1] = fma(rho, fma(w.u, l[3], l[1]), o[1]);
  o[2] = fma(rho, fma(w.v, l[3], l[2]), o[2]);
  o[3] = fma(s * g.gm1inv, l[3], o[3]);
}

template <int FAM, typename T, typename Scatter>
__device__ __forceinline__ void sac_family_adj(const Scatter& S, const T lGp[3][4],
                                               const T lGuv[3][4], T& lpK, T& luK, T& lvK) {
  if constexpr (FAM == 0) af_sac_V_adj<T>(S, lGp, lGuv, lpK, luK, lvK);
  if constexpr (FAM == 1) af_sac_EV_adj<T>(S, lGp, lGuv, lpK, luK, lvK);
  if constexpr (FAM == 2) af_sac_EH_adj<T>(S, lGp, lGuv, lpK, luK, lvK);
  if constexpr (FAM == 3) af_sac_C_adj<T>(S, lGp, lGuv, lpK, luK, lvK);
}


// ---------------------------------------------------------------------------
// Points, reversed: the average update and the space-time Simpson fluxes (Eq.
// af-average-update) as a gather, then the point update (Sec. 6.1 steps 3-4;
// Eq. barsukow-additive).  One thread per point, families by blockIdx.y.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ Prim<T> level_pt(const T* base, size_t ps, int f, size_t id) {
  const T* b = base + (size_t)(4 * f) * ps + id;
  Prim<T> w = {b[0], b[ps], b[2 * ps], b[3 * ps]};
  return w;
}

// lambda^{n+1} as given, in the working precision
template <typename T>
__device__ __forceinline__ T lam_in(const AdjView<T>& v, int plane, size_t id) {
  return (T)v.lin64[plane][id];
}

// Adjoints of the x- and y-fluxes (lex, ley, before the factor dt / (36 h)) that
// the point of family FAM of cell (i, j) enters, and lambda of the point itself;
// also passes lambda of the averages through (family 0, one writer per cell).
// Every load is issued before the first use.
template <int FAM, typename T>
__device__ __forceinline__ void flux_lambda(const AdjView<T>& v, int i, int j, size_t id, T lex[4],
                                            T ley[4], T lpt[4]) {
  const int im = i == 0 ? v.nx - 1 : i - 1, jm = j == 0 ? v.ny - 1 : j - 1;
  const size_t idl = (size_t)j * v.nx + im, idb = (size_t)jm * v.nx + i,
               idlb = (size_t)jm * v.nx + im;
  T c[4], l[4], b[4], lb[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    c[k] = lam_in(v, k, id);
    if (FAM != 2) l[k] = lam_in(v, k, idl);
    if (FAM != 1) b[k] = lam_in(v, k, idb);
    if (FAM == 0) lb[k] = lam_in(v, k, idlb);
    lpt[k] = lam_in(v, 4 + 4 * FAM + k, id);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (FAM == 0) {
      lex[k] = (c[k] - l[k]) + (b[k] - lb[k]);
      ley[k] = (c[k] - b[k]) + (l[k] - lb[k]);
      v.lam[(size_t)(LAM_OUT + k) * v.ps + id] = c[k];
    } else if (FAM == 1) {
      lex[k] = c[k] - l[k];
    } else {
      ley[k] = c[k] - b[k];
    }
  }
}

// o = the share of the fluxes' adjoints that reaches the node value w; lex, ley
// carry the factor dt / (36 h), sc the time and edge-midpoint weights
template <int FAM, typename T>
__device__ __forceinline__ void flux_share(const Prim<T>& w, const Gas<T>& g, const T lex[4],
                                           const T ley[4], T sc, T o[4]) {
  T l[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) o[k] = T(0);
  if (FAM != 2) {
#pragma unroll
    for (int k = 0; k < 4; ++k) l[k] = sc * lex[k];
    flux_x_adj(w, g, l, o);
  }
  if (FAM != 1) {
#pragma unroll
    for (int k = 0; k < 4; ++k) l[k] = sc * ley[k];
    flux_y_adj(w, g, l, o);
  }
}

// Fluxes of the point of family FAM of cell (i, j), reversed: its adjoints at
// sigma = 0 (own node, value wp), 1/2 and 1 (values wh, wf; lambda^{n+1} of the
// point included in the last).
template <int FAM, typename T>
__device__ __forceinline__ void point_fluxes_adj(const AdjView<T>& v, int i, int j, size_t id,
                                                 const Prim<T>& wp, const Prim<T>& wh,
                                                 const Prim<T>& wf, T own[4], T lyh[4], T lyf[4]) {
  T lex[4], ley[4], lpt[4];
  flux_lambda<FAM>(v, i, j, id, lex, ley, lpt);
  const T cst = v.dth / T(36), mid = FAM == 0 ? cst : T(4) * cst;
  flux_share<FAM>(wp, v.gas, lex, ley, mid, own);
  flux_share<FAM>(wh, v.gas, lex, ley, T(4) * mid, lyh);
  flux_share<FAM>(wf, v.gas, lex, ley, mid, lyf);
#pragma unroll
  for (int k = 0; k < 4; ++k) lyf[k] += lpt[k];
}

// sum over the nine nodes of d/d(xi) and d/d(eta) of the Q2 basis times dot[]
template <typename T>
__device__ __forceinline__ void grad_sum(const T dot[9], const T lx[3], const T ly[3],
                                         const T dx[3], const T dy[3], T& gx, T& gy) {
  T rx[3], rl[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    rx[b] = fma(dx[0], dot[3 * b], fma(dx[1], dot[3 * b + 1], dx[2] * dot[3 * b + 2]));
    rl[b] = fma(lx[0], dot[3 * b], fma(lx[1], dot[3 * b + 1], lx[2] * dot[3 * b + 2]));
  }
  gx = fma(ly[0], rx[0], fma(ly[1], rx[1], ly[2] * rx[2]));
  gy = fma(dy[0], rl[0], fma(dy[1], rl[1], dy[2] * rl[2]));
}

// the point of family FAM of cell (i, j), both durations
template <int FAM, typename T>
__device__ __forceinline__ void point_adj(const AdjView<T>& v, int i, int j, size_t id) {
  const size_t ps = v.ps;
  const int nx = v.nx, ny = v.ny;
  constexpr int OX = FAM == 2 ? 1 : 0, OY = FAM == 1 ? 1 : 0;
  const Gas<T>& g = v.gas;
  const Prim<T> wp = level_pt(v.st + 4 * ps, ps, FAM, id);
  auto wplane = [&](int k) {  // time-n values: component k of family f
    return [&v, k](int f) {
      return f < 3 ? v.st + (size_t)(4 + 4 * f + k) * v.ps : v.scr + (size_t)k * v.ps;
    };
  };
  auto node_rec = [&](int f, size_t q) {
    return v.lam + (size_t)(LAM_NODE + 4 * f) * ps + 4 * q;
  };
  T own[4], lyh[4], lyf[4];
  point_fluxes_adj<FAM>(v, i, j, id, wp,
                        level_pt(v.scr + (size_t)SCR_HALF * ps, ps, FAM, id),
                        level_pt(v.sto + 4 * ps, ps, FAM, id), own, lyh, lyf);
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const T th = s == 0 ? T(0.5) * v.dth : v.dth;
    T ly[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) ly[k] = s == 0 ? lyh[k] : lyf[k];
    auto iplane = [&](int k) {
      return [&v, s, k](int f) { return v.scr + (size_t)(SCR_INC + 12 * s + 3 * f + k) * v.ps; };
    };
    // forward recomputation of the foot (Eq. adv-footpoint)
    int c1x, c1y, cfx, cfy;
    T lx1[3], ly1[3], lx[3], lyb[3], dx1[3], dy1[3], dx3[3], dy3[3];
    {
      const T sx = foot_coord<OX>(-th * wp.u, c1x), sy = foot_coord<OY>(-th * wp.v, c1y);
      lagrange3_fma(sx, lx1);
      lagrange3_fma(sy, ly1);
      lagrange3_d(sx, dx1);
      lagrange3_d(sy, dy1);
    }
    const FootNodes n1 = foot_nodes(i + c1x, j + c1y, nx, ny);
    {
      const T u1 = row_sum(n1, lx1, ly1, wplane(1)), v1 = row_sum(n1, lx1, ly1, wplane(2));
      const T sx = foot_coord<OX>(-th * u1, cfx), sy = foot_coord<OY>(-th * v1, cfy);
      lagrange3_fma(sx, lx);
      lagrange3_fma(sy, lyb);
      lagrange3_d(sx, dx3);
      lagrange3_d(sy, dy3);
    }
    const FootNodes nf = foot_nodes(i + cfx, j + cfy, nx, ny);
    T w[9];
#pragma unroll
    for (int m = 0; m < 9; ++m) w[m] = lx[m % 3] * lyb[m / 3];
    const T rft = row_sum(nf, lx, lyb, wplane(0)), pft = row_sum(nf, lx, lyb, wplane(3));
    T lwf[4], ldp = T(0);  // adjoints of W_f and of the interpolated dp (du, dv: lwf[1], lwf[2])
    if (v.variant == 0) {
      const T d2 = row_sum(nf, lx, lyb, iplane(2));
      const T rf = with_ref(g.rho_ref, rft), pf = with_ref(g.p_ref, pft);
      const T igp = T(1) / (g.gamma * pf);
      const T a0 = ly[0] * igp;
      lwf[0] = fma(a0, d2, ly[0]);
      lwf[1] = ly[1];
      lwf[2] = ly[2];
      lwf[3] = fma(-(a0 * d2) * rf, igp * g.gamma, ly[3]);
      ldp = fma(a0, rf, ly[3]);
    } else {
      const T d2 = iplane(2)(FAM)[id];
      const T rp = with_ref(g.rho_ref, wp.r), pp = with_ref(g.p_ref, wp.p);
      const T igp = T(1) / (g.gamma * pp);
      const T a0 = ly[0] * igp;
#pragma unroll
      for (int k = 0; k < 4; ++k) lwf[k] = ly[k];
      // nw.r = wf.r + dp rho_P / (gamma p_P), with the increments at P itself
      add4(v.lam + (size_t)(LAM_INC + 4 * (4 * s + FAM)) * ps + 4 * id, ly[1], ly[2],
           fma(a0, rp, ly[3]), T(0));
      own[0] = fma(a0, d2, own[0]);
      own[3] = fma(-(a0 * d2) * rp, igp * g.gamma, own[3]);
    }
    // adjoint of the foot's local coordinates through the Q2 evaluation there (u
    // and du enter the transported update with the same weight; the increment
    // planes hold their sum)
    T dot[9], gx, gy;
#pragma unroll
    for (int m = 0; m < 9; ++m) {
      const int f = fam_of(m % 3, m / 3);
      const size_t q = nf.n[m / 3 >> 1][m % 3 >> 1];
      T t = fma(wplane(0)(f)[q], lwf[0], wplane(3)(f)[q] * lwf[3]);
      if (v.variant == 0) {
        t = fma(iplane(0)(f)[q], lwf[1], t);
        t = fma(iplane(1)(f)[q], lwf[2], t);
        dot[m] = fma(iplane(2)(f)[q], ldp, t);
      } else {
        t = fma(wplane(1)(f)[q], lwf[1], t);
        dot[m] = fma(wplane(2)(f)[q], lwf[2], t);
      }
    }
    grad_sum(dot, lx, lyb, dx3, dy3, gx, gy);
    // xi = 2 (foot - cell) - 1; the foot moved by df = -th (u1, v1)
    const T lu1 = T(-2) * th * gx, lv1 = T(-2) * th * gy;
    // first Picard stage: (u1, v1) = R_h(u, v) at P + d1
#pragma unroll
    for (int m = 0; m < 9; ++m) {
      const int f = fam_of(m % 3, m / 3);
      const size_t q = n1.n[m / 3 >> 1][m % 3 >> 1];
      dot[m] = fma(wplane(1)(f)[q], lu1, wplane(2)(f)[q] * lv1);
    }
    grad_sum(dot, lx1, ly1, dx1, dy1, gx, gy);
    own[1] = fma(T(-2) * th, gx, own[1]);
    own[2] = fma(T(-2) * th, gy, own[2]);
    // scatter to the nodes of the foot cell and of the first stage's cell (one
    // record update per node when the two cells coincide, the usual case)
    const bool same = c1x == cfx && c1y == cfy;
#pragma unroll
    for (int m = 0; m < 9; ++m) {
      const int f = fam_of(m % 3, m / 3);
      const size_t q = nf.n[m / 3 >> 1][m % 3 >> 1];
      const T wu = w[m] * lwf[1], wv = w[m] * lwf[2];
      T nu = wu, nv = wv;
      if (same) {
        const T w1 = lx1[m % 3] * ly1[m / 3];
        nu = fma(w1, lu1, wu);
        nv = fma(w1, lv1, wv);
      }
      add4_always(node_rec(f, q), w[m] * lwf[0], nu, nv, w[m] * lwf[3]);
      if (v.variant == 0)
        add3_always(v.lam + (size_t)(LAM_INC + 4 * (4 * s + f)) * ps + 4 * q, wu, wv, w[m] * ldp);
    }
    if (!same) {
#pragma unroll
      for (int m = 0; m < 9; ++m) {
        const T w1 = lx1[m % 3] * ly1[m / 3];
        add4(node_rec(fam_of(m % 3, m / 3), n1.n[m / 3 >> 1][m % 3 >> 1]), T(0), w1 * lu1,
             w1 * lv1, T(0));
      }
    }
  }
  add4_always(node_rec(FAM, id), own[0], own[1], own[2], own[3]);
}

template <typename T>
__global__ void __launch_bounds__(REF_THREADS) k_adj_points(const __grid_constant__ AdjView<T> v) {
  pdl_wait();
  const size_t id = (size_t)blockIdx.x * REF_THREADS + threadIdx.x;
  if (id >= (size_t)v.nx * v.ny) return;
  const int j = (int)(id / (unsigned)v.nx), i = (int)(id - (size_t)j * v.nx);
  switch (blockIdx.y) {
    case 0: point_adj<0>(v, i, j, id); break;
    case 1: point_adj<1>(v, i, j, id); break;
    default: point_adj<2>(v, i, j, id); break;
  }
}

// ---------------------------------------------------------------------------
// Acoustic increments (Sec. 6.1 step 1), reversed: Horner in r_s = c tau_s / h,
// freezing c = sqrt(gamma p / rho), Z = rho c, and the transposed stencils.
// ---------------------------------------------------------------------------
// node values (.p, .u, .v) at lattice offset (dx, dy) from the node of family
// FAM of the neighbourhood's centre cell
template <int FAM, typename T>
struct LoadAdjPUV {
  const AdjView<T>* v;
  Nbhd b;
  __device__ __forceinline__ PUV<T> operator()(int dx, int dy) const {
    const int ax = ((FAM == 2 || FAM == 3) ? 1 : 0) + dx, by = ((FAM == 1 || FAM == 3) ? 1 : 0) + dy;
    const Prim<T> w = node_w(*v, fam_of(ax, by), b.at(ax >> 1, by >> 1));
    PUV<T> o = {w.p, w.u, w.v};
    return o;
  }
};

// adds (lp, lu, lv) to the record of the node at lattice offset (dx, dy).
// The warp is one row of consecutive nodes (lane = x offset); `act` holds the
// lanes taking part.  pair() takes a member (dx, dy), dx > 0, and its mirror
// (-dx, dy): the mirror's target seen from lane k + delta (delta = the cell
// distance between the two targets) is the member's target seen from lane k,
// so lane k adds lane k + delta's mirror values to its own and makes one
// record update for both; a mirror value whose lane k - delta is not taking
// part is added on its own.
template <int FAM, typename T>
struct ScatterAdj {
  T* lam;
  size_t ps;
  Nbhd b;
  unsigned act;
  __device__ __forceinline__ T* rec(int ax, int by) const {
    return lam + (size_t)(LAM_NODE + 4 * fam_of(ax, by)) * ps + 4 * b.at(ax >> 1, by >> 1);
  }
  __device__ __forceinline__ void operator()(int dx, int dy, T lp, T lu, T lv) const {
    constexpr int ox = (FAM == 2 || FAM == 3) ? 1 : 0, oy = (FAM == 1 || FAM == 3) ? 1 : 0;
    add4_always(rec(ox + dx, oy + dy), T(0), lu, lv, lp);
  }
  __device__ __forceinline__ void pair(int dx, int dy, T lp, T lu, T lv, T mp, T mu,
                                       T mv) const {
    constexpr int ox = (FAM == 2 || FAM == 3) ? 1 : 0, oy = (FAM == 1 || FAM == 3) ? 1 : 0;
    const int ax = ox + dx, am = ox - dx, by = oy + dy;
    const int delta = (ax >> 1) - (am >> 1);  // 1 or 2 (compile time once inlined)
    const int lane = threadIdx.x & 31;
    const T sp = __shfl_down_sync(act, mp, delta), su = __shfl_down_sync(act, mu, delta),
            sv = __shfl_down_sync(act, mv, delta);
    const bool take = lane + delta < 32 && ((act >> (lane + delta)) & 1u);
    const bool alone = lane < delta || !((act >> (lane - delta)) & 1u);
    add4_always(rec(ax, by), T(0), take ? lu + su : lu, take ? lv + sv : lv, take ? lp + sp : lp);
    if (alone) add4_always(rec(am, by), T(0), mu, mv, mp);
  }
  // members (2, dy), (-2, dy), (0, dy) of a family whose own column is even:
  // three consecutive nodes of one row, the right one lane k + 1's centre, the
  // left one lane k - 1's.  Each lane updates its centre with its neighbours'
  // right and left values, and its own right (left) value alone when lane
  // k + 1 (k - 1) is not taking part.
  __device__ __forceinline__ void triple(int dy, T rp, T ru, T rv, T lp, T lu, T lv, T cp, T cu,
                                         T cv) const {
    static_assert(FAM == 0 || FAM == 1, "the node's own column is even");
    constexpr int oy = FAM == 1 ? 1 : 0;
    const int by = oy + dy;
    const int lane = threadIdx.x & 31;
    const T ip = __shfl_up_sync(act, rp, 1), iu = __shfl_up_sync(act, ru, 1),
            iv = __shfl_up_sync(act, rv, 1);  // lane k - 1's right values
    const T jp = __shfl_down_sync(act, lp, 1), ju = __shfl_down_sync(act, lu, 1),
            jv = __shfl_down_sync(act, lv, 1);  // lane k + 1's left values
    const bool from_l = lane >= 1 && ((act >> (lane - 1)) & 1u);
    const bool from_r = lane <= 30 && ((act >> (lane + 1)) & 1u);
    T p = cp, u = cu, w = cv;
    if (from_l) {
      p += ip;
      u += iu;
      w += iv;
    }
    if (from_r) {
      p += jp;
      u += ju;
      w += jv;
    }
    add4_always(rec(0, by), T(0), u, w, p);
    if (!from_r) add4_always(rec(2, by), T(0), ru, rv, rp);
    if (!from_l) add4_always(rec(-2, by), T(0), lu, lv, lp);
  }
};

// `row`: the lanes of the calling warp (one row of 32 consecutive nodes) inside
// the grid
template <int FAM, typename T>
__device__ __forceinline__ void acoustic_adj(const AdjView<T>& v, int i, int j, unsigned row) {
  const size_t ps = v.ps, id = (size_t)j * v.nx + i;
  T ld[2][3];
  bool any = false;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    T* rec = v.lam + (size_t)(LAM_INC + 4 * (4 * s + FAM)) * ps + 4 * id;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ld[s][k] = rec[k];
      any = any || ld[s][k] != T(0);
    }
  }
  // the lanes of the row that have work: they take part in the merged scatter
  const unsigned act = __ballot_sync(row, any);
  if (!any) return;
#pragma unroll
  for (int s = 0; s < 2; ++s) zero4(v.lam + (size_t)(LAM_INC + 4 * (4 * s + FAM)) * ps + 4 * id);
  const Prim<T> wk = node_w(v, FAM, id);
  const T rk = with_ref(v.gas.rho_ref, wk.r), pk = with_ref(v.gas.p_ref, wk.p);
  T c, Z, Zinv;
  freeze(v.gas.gamma, rk, pk, c, Z, Zinv);
  const T dth = v.dth;
  const T r1 = c * dth;
  T Gp[3][4], Guv[3][4];
  const Nbhd nb = nbhd(i, j, v.nx, v.ny);
  const LoadAdjPUV<FAM, T> ldr = {&v, nb};
  sac_family<FAM, T>(ldr, wk.p, wk.u, wk.v, Gp, Guv);
  // polynomial coefficients c_o[q] (q = 1..4 stored at 0..3), as in acoustic_node
  T co[3][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    co[2][q] = fma(Z, Guv[0][q], Gp[0][q]);     // dp
    co[0][q] = fma(Zinv, Gp[1][q], Guv[1][q]);  // du
    co[1][q] = fma(Zinv, Gp[2][q], Guv[2][q]);  // dv
  }
  T lco[3][4], lr1 = T(0);
  {
    // powers of r_s = r1 / 2, r1; d(delta_o)/dr1 = sum_q q r^{q-1} co[o][q], times
    // 1/2 for s = 0
    T pw[2][5];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      pw[s][0] = T(1);
      pw[s][1] = s == 0 ? T(0.5) * r1 : r1;
#pragma unroll
      for (int q = 2; q <= 4; ++q) pw[s][q] = pw[s][q - 1] * pw[s][1];
    }
#pragma unroll
    for (int o = 0; o < 3; ++o) {
#pragma unroll
      for (int q = 1; q <= 4; ++q) lco[o][q - 1] = fma(pw[0][q], ld[0][o], pw[1][q] * ld[1][o]);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const T r = pw[s][1];
        const T dr = fma(r, fma(r, fma(r, T(4) * co[o][3], T(3) * co[o][2]), T(2) * co[o][1]),
                         co[o][0]);
        lr1 = fma(s == 0 ? T(0.5) * dr : dr, ld[s][o], lr1);
      }
    }
  }
  T lGp[3][4], lGuv[3][4], lZ = T(0), lZinv = T(0);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    lGp[0][q] = lco[2][q];
    lGuv[0][q] = Z * lco[2][q];
    lZ = fma(Guv[0][q], lco[2][q], lZ);
    lGp[1][q] = Zinv * lco[0][q];
    lGuv[1][q] = lco[0][q];
    lZinv = fma(Gp[1][q], lco[0][q], lZinv);
    lGp[2][q] = Zinv * lco[1][q];
    lGuv[2][q] = lco[1][q];
    lZinv = fma(Gp[2][q], lco[1][q], lZinv);
  }
  lZ = fma(-lZinv * Zinv, Zinv, lZ);
  // c^2 = gamma p / rho: dc/drho = -c / (2 rho), dc/dp = c / (2 p) = gamma / (2 Z)
  const T lc = fma(dth, lr1, rk * lZ), hc = T(0.5) * lc;
  const T lrho = fma(c, lZ, -hc * c / rk);
  const T lp = hc * (v.gas.gamma * Zinv);
  T lpK = T(0), luK = T(0), lvK = T(0);
  const ScatterAdj<FAM, T> S = {v.lam, v.ps, nb, act};
  sac_family_adj<FAM, T>(S, lGp, lGuv, lpK, luK, lvK);
  add4(v.lam + (size_t)(LAM_NODE + 4 * FAM) * ps + 4 * id, lrho, luK, lvK, lp + lpK);
}

// Blocks of the acoustic adjoint: BY rows of 32 consecutive nodes.  FP32 waits on
// scattered loads and atomics, and the vertex family spills below 96 registers: 128
// threads, five blocks per SM (adjoint step at 2048^2 2.89 ms; three of 256 threads at
// 80 registers 2.94, two at 128 2.98, four of 128 or of 192 2.95 and 2.93; measured with
// one reciprocal root for the freezing, with IEEE operations the chosen one takes 2.98).  FP64 is bound
// by its arithmetic unit and would spill: two warps, registers as needed.
template <typename T>
struct AdjBlock {
  static constexpr int BY = sizeof(T) == 4 ? 4 : 2, MINB = sizeof(T) == 4 ? 5 : 1;
};

// its blocks per family: 32 columns x BY rows each
template <typename T>
inline unsigned adj_acoustic_blocks(int nx, int ny) {
  constexpr int BY = AdjBlock<T>::BY;
  return (unsigned)((size_t)((nx + 31) / 32) * ((ny + BY - 1) / BY));
}

// Blocks of one family along blockIdx.x, row by row (the limit of 65535 on a grid's
// other dimensions is no limit on the rows); the families by blockIdx.y.
template <typename T>
__global__ void __launch_bounds__(32 * AdjBlock<T>::BY, AdjBlock<T>::MINB)
    k_adj_acoustic(const __grid_constant__ AdjView<T> v) {
  pdl_wait();
  // a warp is one row of 32 consecutive nodes (blockDim.x == 32)
  const unsigned cols = (unsigned)(v.nx + 31) / 32, br = blockIdx.x / cols;
  const int i = (int)((blockIdx.x - br * cols) * 32 + threadIdx.x);
  const int j = (int)(br * AdjBlock<T>::BY + threadIdx.y);
  const unsigned row = __ballot_sync(0xffffffffu, i < v.nx && j < v.ny);
  if (i >= v.nx || j >= v.ny) return;
  switch (blockIdx.y) {
    case 0: acoustic_adj<0>(v, i, j, row); break;
    case 1: acoustic_adj<1>(v, i, j, row); break;
    case 2: acoustic_adj<2>(v, i, j, row); break;
    default: acoustic_adj<3>(v, i, j, row); break;
  }
}

// ---------------------------------------------------------------------------
// Centre recovery (Eq. center-node), reversed, in two parts: k_adj_center turns
// each cell's centre adjoint lambda_W into lambda_U (the adjoint of the
// recovered conserved centre), adds its 9/4 share to the cell average's lambda
// and stores lambda_U; k_adj_out then gives every vertex and edge node the
// -1/16 and -1/4 shares of the cells around it (a gather: four cells for a
// vertex, two for an edge, no atomics) before writing lambda^n out.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(REF_THREADS) k_adj_center(const __grid_constant__ AdjView<T> v) {
  pdl_wait();
  const size_t id = (size_t)blockIdx.x * REF_THREADS + threadIdx.x, ps = v.ps;
  if (id >= (size_t)v.nx * v.ny) return;
  T* lc = v.lam + (size_t)(LAM_NODE + 12) * ps + 4 * id;  // the centre node's record
  const T lw[4] = {lc[0], lc[1], lc[2], lc[3]};
  T lU[4] = {T(0), T(0), T(0), T(0)};
  if (lw[0] != T(0) || lw[1] != T(0) || lw[2] != T(0) || lw[3] != T(0)) {
    zero4(lc);
    const Gas<T>& g = v.gas;
    // the recovered centre (rho~, u, v, p~) is W(U_c); lambda_U = (dW/dU)^T lambda_W
    const T rho = with_ref(g.rho_ref, v.scr[id]), u = v.scr[ps + id], w = v.scr[2 * ps + id];
    const T ri = T(1) / rho, gl = g.gm1 * lw[3];
    const T a1 = ri * lw[1], a2 = ri * lw[2];
    lU[0] = fma(gl, T(0.5) * fma(u, u, w * w), fma(-w, a2, fma(-u, a1, lw[0])));
    lU[1] = fma(-u, gl, a1);
    lU[2] = fma(-w, gl, a2);
    lU[3] = gl;
    // U_c = 9/4 Ubar - 1/16 sum_corners U(W) - 1/4 sum_edges U(W); the
    // average of this cell has no other writer in this kernel
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      T* o = v.lam + (size_t)(LAM_OUT + k) * ps + id;
      *o = fma(T(2.25), lU[k], *o);
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) v.lam[(size_t)(LAM_LU + k) * ps + id] = lU[k];
}

// ---------------------------------------------------------------------------
// Fused reverse sweep of a tile (FP32 modes).  fused_tile<..., ADJ> leaves the
// tile's time-n nodes W and the increments D of both durations in shared
// memory.  For each owned point: the adjoint of the space-time Simpson fluxes
// it enters (gathered from the averages' lambda, point_fluxes_adj), then the
// adjoint of its point update for both durations (as k_adj_points) with the
// forward values taken from shared memory and the foot traced as the fused
// step traces it (displacements clamped to one cell).  Results go to the node
// and increment records (float4 atomics); the averages' lambda passes through.
// ---------------------------------------------------------------------------
template <int TX, int TY, int NT>
__device__ __forceinline__ void tile_reverse(const StepArgs<float>& a, const AdjView<float>& v,
                                             const float4* W, const float* D, int i0, int j0) {
  using G = FusedGeom<TX, TY>;
  constexpr int CW = G::CW, WPL = G::WPL, DCW = G::DCW, DPL = G::DPL;
  const int nx = a.nx, ny = a.ny;
  const size_t ps = v.ps;
  const Gas<float> gas = a.gas;
  const float th_full = a.dt / a.h;
  // (a warp is consecutive points of whole rows of one family, and a round is taken
  // or left by all its lanes)
  static_assert(32 % TX == 0 && (TX * TY) % 32 == 0, "a warp holds rows of one family");
  const int lane = threadIdx.x & 31;
  for (int t = threadIdx.x; t < 3 * TX * TY; t += NT) {
    const int fam = t / (TX * TY), u = t - fam * (TX * TY);
    const int px = u % TX, py = u / TX;
    const int gi = i0 + px, gj = j0 + py;
    // lanes of the warp inside the grid (every lane of the warp is here)
    const unsigned mask = __ballot_sync(0xffffffffu, gi < nx && gj < ny);
    if (gi >= nx || gj >= ny) continue;
    const size_t id = (size_t)gj * nx + gi;
    // ---- fluxes (Eq. af-average-update), reversed ----
    const int wcP = (py + 2) * CW + (px + 2);
    const float4 wp = W[fam * WPL + wcP];
    float o0[4], lyh[4], lyf[4];  // sigma = 0 (own node), 1/2 and 1 (the point)
    {
      float* const* hp = a.half[fam];
      float* const* np = a.out.pt[fam];
      const Prim<float> wh = {hp[0][id], hp[1][id], hp[2][id], hp[3][id]};
      const Prim<float> wf = {np[0][id], np[1][id], np[2][id], np[3][id]};
      if (fam == 0)
        point_fluxes_adj<0>(v, gi, gj, id, prim4(wp), wh, wf, o0, lyh, lyf);
      else if (fam == 1)
        point_fluxes_adj<1>(v, gi, gj, id, prim4(wp), wh, wf, o0, lyh, lyf);
      else
        point_fluxes_adj<2>(v, gi, gj, id, prim4(wp), wh, wf, o0, lyh, lyf);
    }
    // ---- point update (Sec. 6.1 steps 3-4), reversed, both durations ----
    const int ox = fam == 2 ? 1 : 0, oy = fam == 1 ? 1 : 0;
    float luP = 0.f, lvP = 0.f, lrP = 0.f, lpP = 0.f;
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
      const float th = s == 0 ? 0.5f * th_full : th_full;
      const float* Ds = D + s * 12 * DPL;
      float ly[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) ly[k] = s == 0 ? lyh[k] : lyf[k];
      // forward: the two Picard stages as the fused step traces them
      // (shared node records are (u, v, rho~, p~))
      const float d1x = clamp1(-th * wp.x), d1y = clamp1(-th * wp.y);
      float lx1[3], ly1[3];
      const int ix1 = foot_axis(ox, d1x, lx1), iy1 = foot_axis(oy, d1y, ly1);
      const int c1 = wcP + iy1 * CW + ix1;
      float4 n[9];
      load_cell<CW, WPL>(W, c1, n);
      const float u1 = AF_Q2(n, x, lx1, ly1), v1 = AF_Q2(n, y, lx1, ly1);
      const float dfx = clamp1(-th * u1), dfy = clamp1(-th * v1);
      float lx[3], lyb[3];
      const int ix = foot_axis(ox, dfx, lx), iy = foot_axis(oy, dfy, lyb);
      const int c2 = wcP + iy * CW + ix;
      if (c2 != c1) load_cell<CW, WPL>(W, c2, n);
      const float rft = AF_Q2(n, z, lx, lyb), pft = AF_Q2(n, w, lx, lyb);
      // local coordinates of the foot and of the first stage
      float dx3[3], dy3[3], dx31[3], dy31[3];
      {
        const float fx = fmaf(0.5f, (float)ox, dfx), fy = fmaf(0.5f, (float)oy, dfy);
        lagrange3_d(fmaf(2.f, fx - floorf(fx), -1.f), dx3);
        lagrange3_d(fmaf(2.f, fy - floorf(fy), -1.f), dy3);
        const float gx = fmaf(0.5f, (float)ox, d1x), gy = fmaf(0.5f, (float)oy, d1y);
        lagrange3_d(fmaf(2.f, gx - floorf(gx), -1.f), dx31);
        lagrange3_d(fmaf(2.f, gy - floorf(gy), -1.f), dy31);
      }
      const int dcf = (py + 1 + iy) * DCW + (px + 1 + ix);  // D cell of the foot cell
      float lwf[4], ld[3];  // adjoints of W at the foot and of the interpolated increments
      if (a.variant == 0) {
        const float d2 = q2_eval<DCW>(Ds + 2 * DPL, Ds + 5 * DPL, Ds + 8 * DPL, Ds + 11 * DPL,
                                      dcf, lx, lyb);
        // (fast reciprocals, as the forward closure's division: with IEEE divisions and
        // roots throughout the sweep the errors against FP64 are the same to 1%, 1024^2
        // takes 809 us instead of 790)
        const float rf = gas.rho_ref + rft, pf = gas.p_ref + pft;
        const float igp = __fdividef(1.f, gas.gamma * pf), ipf = __fdividef(1.f, pf);
        lwf[0] = ly[0] * fmaf(d2, igp, 1.f);
        lwf[1] = ly[1];
        lwf[2] = ly[2];
        lwf[3] = ly[3] - ly[0] * d2 * rf * igp * ipf;
        ld[0] = ly[1];
        ld[1] = ly[2];
        ld[2] = fmaf(ly[0] * rf, igp, ly[3]);
      } else {
        const int dcp = (py + 1) * DCW + (px + 1);
        const float d2 = Ds[(fam * 3 + 2) * DPL + dcp];
        const float rp = gas.rho_ref + wp.z, pp = gas.p_ref + wp.w;
        const float igp = __fdividef(1.f, gas.gamma * pp), ipp = __fdividef(1.f, pp);
#pragma unroll
        for (int k = 0; k < 4; ++k) lwf[k] = ly[k];
        // rho = rho_f + dp rho_P / (gamma p_P), with the increments at P itself
        add4(v.lam + (size_t)(LAM_INC + 4 * (4 * s + fam)) * ps + 4 * id, ly[1], ly[2],
             fmaf(ly[0] * rp, igp, ly[3]), 0.f);
        lrP += ly[0] * d2 * igp;
        lpP += -ly[0] * d2 * rp * igp * ipp;
        ld[0] = ld[1] = ld[2] = 0.f;
      }
      // adjoint of the foot's local coordinates.  D holds (u + du, v + dv) and dp;
      // u and du enter the transported update with the same weight.
      float lxi = 0.f, leta = 0.f;
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int m = 3 * b + q, fn = fam_of(q, b);
          float dot;
          if (a.variant == 0) {
            const int dn = dcf + (b >> 1) * DCW + (q >> 1);
            const float2 uv = reinterpret_cast<const float2*>(Ds + fn * 3 * DPL)[dn];
            dot = n[m].z * lwf[0] + uv.x * lwf[1] + uv.y * lwf[2] + n[m].w * lwf[3] +
                  Ds[(fn * 3 + 2) * DPL + dn] * ld[2];
          } else {
            dot = n[m].z * lwf[0] + n[m].x * lwf[1] + n[m].y * lwf[2] + n[m].w * lwf[3];
          }
          lxi += dx3[q] * lyb[b] * dot;
          leta += lx[q] * dy3[b] * dot;
        }
      // xi = 2 (foot - cell) - 1; the foot moved by df = -th (u1, v1)
      const float lu1 = -th * (2.f * lxi), lv1 = -th * (2.f * leta);
      // first Picard stage: (u1, v1) = R_h(u, v) at P + d1
      if (c2 != c1) load_cell<CW, WPL>(W, c1, n);
      float lxi1 = 0.f, leta1 = 0.f;
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int m = 3 * b + q;
          const float dot = n[m].x * lu1 + n[m].y * lv1;
          lxi1 += dx31[q] * ly1[b] * dot;
          leta1 += lx1[q] * dy31[b] * dot;
        }
      luP += -th * (2.f * lxi1);
      lvP += -th * (2.f * leta1);
      // scatter to the foot cell's nodes (and the first stage's, merged when
      // both use the same cell).  When the right-hand neighbour lane (the next
      // point of the row) has its foot at the same offset, its first node
      // column is this lane's last: it hands those contributions over and this
      // lane adds them with its own (one record update instead of two).
      const bool same = c1 == c2;
      // wrapped cells of the foot cell's 2 x 2 block of node cells
      const int col0 = wrapc(gi + ix, nx), col1 = col0 + 1 == nx ? 0 : col0 + 1;
      const size_t row0 = (size_t)wrapc(gj + iy, ny) * nx;
      const size_t row1 = (row0 + nx == (size_t)ny * nx) ? 0 : row0 + nx;
      const int key = (ix + 2) + 8 * (iy + 2);
      const int lkey = __shfl_up_sync(mask, key, 1), rkey = __shfl_down_sync(mask, key, 1);
      const bool give = px > 0 && ((mask >> (lane - 1)) & 1u) && lkey == key;
      const bool take = px < TX - 1 && ((mask >> (lane + 1)) & 1u) && rkey == key;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        float nd[3][4], ic[3][3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float wgt = lx[q] * lyb[b], w1 = same ? lx1[q] * ly1[b] : 0.f;
          nd[q][0] = wgt * lwf[0];
          nd[q][1] = fmaf(w1, lu1, wgt * lwf[1]);
          nd[q][2] = fmaf(w1, lv1, wgt * lwf[2]);
          nd[q][3] = wgt * lwf[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) ic[q][k] = wgt * ld[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float r = __shfl_down_sync(mask, nd[0][k], 1);
          if (take) nd[2][k] += r;
        }
        if (a.variant == 0) {
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const float r = __shfl_down_sync(mask, ic[0][k], 1);
            if (take) ic[2][k] += r;
          }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          if (q == 0 && give) continue;
          const int fn = fam_of(q, b);
          const size_t cell = (b >> 1 ? row1 : row0) + (q >> 1 ? col1 : col0);
          float* nr = v.lam + (size_t)(LAM_NODE + 4 * fn) * ps + 4 * cell;
          atomicAdd(reinterpret_cast<float4*>(nr),
                    make_float4(nd[q][0], nd[q][1], nd[q][2], nd[q][3]));
          if (a.variant == 0) {
            float* ir = v.lam + (size_t)(LAM_INC + 4 * (4 * s + fn)) * ps + 4 * cell;
            atomicAdd(reinterpret_cast<float4*>(ir),
                      make_float4(ic[q][0], ic[q][1], ic[q][2], 0.f));
          }
        }
      }
      if (!same) {
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float w1 = lx1[q] * ly1[b];
            add4(v.lam + (size_t)(LAM_NODE + 4 * fam_of(q, b)) * ps +
                     4 * cell_id(v, gi + ix1 + (q >> 1), gj + iy1 + (b >> 1)),
                 0.f, w1 * lu1, w1 * lv1, 0.f);
          }
      }
    }
    add4(v.lam + (size_t)(LAM_NODE + 4 * fam) * ps + 4 * id, o0[0] + lrP, o0[1] + luP, o0[2] + lvP,
         o0[3] + lpP);
  }
}

// The fused reverse sweep, one CTA per tile of TX x TY cells (any grid).
template <int TX, int TY, int NT, int MINB, bool COMP>
__global__ void __launch_bounds__(NT, MINB)
    k_fused_adj(const __grid_constant__ StepArgs<float> a, const __grid_constant__ AdjView<float> v) {
  using G = FusedGeom<TX, TY>;
  extern __shared__ __align__(16) float4 smem4[];
  pdl_wait();
  PipeCtx none = {nullptr, 0u, 0u, 0, 0u};
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  fused_tile<TX, TY, NT, COMP, false, false, true>(a, none, i0, j0, -1, -1, false);
  tile_reverse<TX, TY, NT>(a, v, smem4, reinterpret_cast<const float*>(smem4 + 4 * G::WPL), i0,
                           j0);
}

template <int TX, int TY, int NT, int MINB, bool COMP>
inline cudaError_t launch_adj_tiles(cudaStream_t s, const StepArgs<float>& a,
                                    const AdjView<float>& v) {
  using G = FusedGeom<TX, TY>;
  constexpr auto kern = k_fused_adj<TX, TY, NT, MINB, COMP>;
  const cudaError_t e = allow_smem<kern>(G::SMEM);
  if (e != cudaSuccess) return e;
  // (the first kernel of an adjoint step: launched when the stream's work is done)
  return launch_kernel(false, kern, dim3((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY), NT, G::SMEM,
                       s, a, v);
}

// Tile geometries of the fused reverse sweep, chosen as the step's (STEP_GEOMS):
// the least (waves x measured time of one wave, FP32_COMP, GB300).  Two CTAs of
// 256 threads share an SM on 32 x 8 tiles: one recomputes its step (FP32 issue)
// while the other waits on its scatter, which makes up for the larger halo at
// every size (adjoint step at 1024^2: one CTA of 32 x 16 tiles 840 us, persistent
// pipelined 32 x 32 tiles 804, this 777; at 2048^2 2.94 ms against 2.97 pipelined,
// 3.17 before).  Adjoint step, 32 x 32 tiles -> chosen: 64^2 116 -> 46 us, 128^2
// 118 -> 54, 192^2 119 -> 66, 256^2 123 -> 79; 1021 x 1024, which had no fused sweep,
// 1.69 -> 0.79 ms.
enum { ADJ_8x8, ADJ_16x8, ADJ_16x16, ADJ_32x8, ADJ_32x24, N_ADJ_GEOMS };
struct AdjGeometry {
  int tx, ty;
  int per_sm;      // resident CTAs per SM
  float us, fill;  // time of one wave, and once per sweep
};
constexpr AdjGeometry ADJ_GEOMS[N_ADJ_GEOMS] = {{8, 8, 1, 15.f, 0.f},
                                                {16, 8, 1, 18.f, 0.f},
                                                {16, 16, 1, 30.f, 0.f},
                                                {32, 8, 2, 34.6f, 12.f},
                                                {32, 24, 1, 72.f, 0.f}};

inline int choose_adj_geometry(const StepArgs<float>& a, int sms) {
  int best = ADJ_32x8;
  float best_us = 1e30f;
  for (int g = 0; g < N_ADJ_GEOMS; ++g) {
    const AdjGeometry& q = ADJ_GEOMS[g];
    if (!tile_rows_fit(a.ny, q.ty)) continue;
    const int64_t tiles = (int64_t)((a.nx + q.tx - 1) / q.tx) * ((a.ny + q.ty - 1) / q.ty);
    const int64_t wave = (int64_t)sms * q.per_sm;
    const float us = (float)((tiles + wave - 1) / wave) * q.us + q.fill;
    if (us < best_us) {
      best_us = us;
      best = g;
    }
  }
  return best;
}

// The fused reverse sweep on one CTA per tile (af_adj_tiles.cu).
template <bool COMP>
cudaError_t launch_adj_tiles_geom(int geom, cudaStream_t s, const StepArgs<float>& a,
                             const AdjView<float>& v);

// lambda^n out: the averages' planes and the point families' node records into
// sixteen FP64 planes
template <typename T>
struct AdjOut {
  double* dst[16];
};

template <typename T>
__global__ void k_adj_out(const __grid_constant__ AdjView<T> v,
                          const __grid_constant__ AdjOut<T> o, size_t n) {
  pdl_wait();
  const size_t ps = v.ps;
  const Gas<T>& g = v.gas;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (size_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int k = 0; k < 4; ++k) o.dst[k][t] = (double)v.lam[(size_t)(LAM_OUT + k) * ps + t];
    // lambda_U of the cells around this cell's vertex (i, j): (i, j), (i-1, j),
    // (i, j-1), (i-1, j-1); the x-edge (i+1/2, j) lies in (i, j) and (i, j-1),
    // the y-edge (i, j+1/2) in (i, j) and (i-1, j)
    const int j = (int)(t / (size_t)v.nx), i = (int)(t - (size_t)j * v.nx);
    const size_t il = (size_t)j * v.nx + wrapc(i - 1, v.nx);
    const size_t jb = (size_t)wrapc(j - 1, v.ny) * v.nx;
    const size_t ib = jb + i, ilb = jb + wrapc(i - 1, v.nx);
    T lc[4], ll[4], lb[4], llb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const T* pl = v.lam + (size_t)(LAM_LU + k) * ps;
      lc[k] = pl[t];
      ll[k] = pl[il];
      lb[k] = pl[ib];
      llb[k] = pl[ilb];
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      T* rec = v.lam + (size_t)(LAM_NODE + 4 * f) * ps + 4 * t;
      T r[4] = {rec[0], rec[1], rec[2], rec[3]}, sum[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        sum[k] = f == 0 ? (lc[k] + ll[k]) + (lb[k] + llb[k]) : (f == 1 ? lc[k] + ll[k] : lc[k] + lb[k]);
      dcons_dprim_T(node_w(v, f, t), g, sum, f == 0 ? T(-0.0625) : T(-0.25), r);
#pragma unroll
      for (int k = 0; k < 4; ++k) o.dst[4 + 4 * f + k][t] = (double)r[k];
      zero4(rec);
    }
  }
}

}  // namespace af
