// af_fc.cuh -- foot-centred exact frozen acoustic point update (Appendix C),
// FP64 only: an analytical reference variant of the point update, not a hot
// path (the paper measures it at about 1000x the cost of the node-centred one).
//
// For a target point P and a duration tau the convective foot F comes from the
// same two Picard stages as the transported update; the acoustic state is
// frozen at F (W_* = R_h W(F), c_*, Z_* = rho_* c_*; Eq. fc-foot-freeze) and the
// disk of radius R = c_* tau is centred at F.  Under the compact footprint
// condition |F - P|_x + R < h/2, |F - P|_y + R < h/2 (Eq. fc-half-footprint)
// the disk is cut only by the grid lines through P: a vertex disk into the four
// cells around P, an edge disk into the two cells beside the edge.
//
// The exact solution of frozen linear acoustics (u_t + c grad pi = 0,
// pi_t + c div u = 0, pi = p / Z_*) at the centre of the disk, for continuous
// piecewise-Q2 data in monomials about F (units of h), is
//   pi(F) = sum_frag sum_ab r^q [ P_ab E_ab - a U_ab m_{a-1,b} - b V_ab m_{a,b-1} ] / 4pi
//   u(F)  = u_0(F) + sum_frag sum_ab { r^q [ -a P_ab m_{a-1,b} + a U_ab m_ab
//             + a V_ab m_{a-1,b+1} ] + a U_ab h_ab + a V_ab h_{a-1,b+1} } / 4pi
//   v(F)  = v_0(F) + (the same with the roles of the axes exchanged)
// with q = a + b, r = R/h, and for each fragment (scaled to the unit disk) its
// area moments m_ij = int xi^i eta^j Psi (Psi = 2 (1 - |w|^2)^{-1/2}, the
// projected-sphere weight), its radius derivative E_ab = r^-q d/dr (r^{q+1} m_ab)
// and its history h_ij = int_0^r s^{q-1} m_ij(s) ds (Eq. fc-moment-families).
//
// The fragment of a cell is written in the frame reflected so that the cell lies
// at xi', eta' >= lam', mu' (its near corner at P): every cell then runs the same
// code, its region assembled by inclusion-exclusion (Eq. fc-role-rows) from the
// full disk (closed form), the single caps {xi >= a}, {eta >= b} (polynomials in
// a, b) and the double cap {xi >= a, eta >= b}, with reflection signs (-1)^i,
// (-1)^j.  The histories scale as h_ij = r^q hhat_ij and only enter added to the
// area moments of the same index: g_ij = m_ij + hhat_ij.
//
// The double cap is sliced into circles of projected radius p around F: on each
// circle the cap is one arc, from (sqrt(p^2 - b^2), b) to (a, sqrt(p^2 - a^2)),
// whose moments B_ij = int x^i y^j dphi are closed forms in the end points, and
//   m_ij = 2 int p B_ij / sqrt(1 - p^2) dp,  hhat_ij = 2 int sqrt(1 - p^2) B_ij / p dp
// over p in [sqrt(a^2 + b^2), 1] by a tanh-sinh rule (square-root singularities
// at both ends; a cut line close to F makes the arc vary on the scale of the
// offset, which the rule's endpoint clustering resolves).
//
// Work split.  The rule's nodes are the cost (FP64 rate: about 180 operations a
// node, 120 nodes, two durations per vertex), so four lanes share each
// (vertex, duration): a quarter of the nodes each, two shuffle rounds to add them
// up, then one of the four cells each.  An edge point's two cells take a lane
// each.  One thread per point with the whole rule in it ran 15.9 ms at 64^2
// whatever the grid (16 blocks, 129 serial nodes with the arc's sines, powers and
// the rule's own exponentials recomputed at each, moments in local memory); this
// form takes a step from 16.9 to 0.67 ms at 64^2 and from 17.1 to 1.62 ms at 128^2.
#pragma once

#include "af_ref_kernels.cuh"

namespace af {
namespace fc {

constexpr double PI = 3.14159265358979323846;

// Moments of a region of the unit disk: area moments m_ij and radius derivatives
// e_ij = r^-q d/dr (r^{q+1} m_ij) for i, j <= 2, and g_ij = m_ij + hhat_ij for the
// indices of contract() (1 <= i + j <= 3, (2,2), (1,3), (3,1)).
struct Moments {
  double m[3][3], e[3][3], g[4][4];
};
__host__ __device__ constexpr bool has_g(int i, int j) {
  return i + j >= 1 && (i + j <= 3 || (i + j == 4 && i != 0 && j != 0));
}

// (1 - a^n), 2 J_j a^{i+1} (1 - a^2)^{j/2} ... of a single cap {xi >= a}, 0 <= a:
// slicing at fixed xi, the chord carries int eta^j Psi d eta = 2 (1 - xi^2)^{j/2} J_j,
// J_0 = pi, J_2 = pi/2 (odd j: 0), so
//   m_i0 = 2 pi (1 - a^{i+1}) / (i+1),
//   m_i2 = pi [(1 - a^{i+1}) / (i+1) - (1 - a^{i+3}) / (i+3)],
// and r d/dr of m(a = d/r) is a 2 J_j a^i (1 - a^2)^{j/2}; the history is the same
// polynomial integrated over the radii s >= d.  Adds c times the cap, reflected
// in its axis if `refl`, to G; AXIS 1 exchanges the roles of xi and eta.
template <int AXIS>
__device__ __forceinline__ void add_single(Moments& G, double c, double a, bool refl) {
  if (!(a < 1.0)) return;
  double pw[6];
  pw[0] = 1.0;
#pragma unroll
  for (int k = 1; k < 6; ++k) pw[k] = pw[k - 1] * a;
  const double oma = 1.0 - a;
#pragma unroll
  for (int j = 0; j <= 2; j += 2)
#pragma unroll
    for (int i = 0; i <= 3; ++i) {
      if (j == 2 && i == 3) continue;
      const int q = i + j;
      const double i1 = 1.0 / (i + 1), i3 = 1.0 / (i + 3);
      double m, hh = 0.0;
      if (j == 0) {
        m = 2.0 * PI * i1 * (1.0 - pw[i + 1]);
        if (i > 0) hh = 2.0 * PI * i1 * fma(-pw[i], oma, (1.0 - pw[i]) * (1.0 / i));
      } else {
        m = PI * fma(-i3, 1.0 - pw[i + 3], i1 * (1.0 - pw[i + 1]));
        hh = PI * fma((i1 - i3) * (1.0 / q), 1.0 - pw[q],
                      oma * fma(i3, pw[i + 2], -i1 * pw[i + 1]));
      }
      const double cc = (refl && (i & 1)) ? -c : c;
      const int x = AXIS == 0 ? i : j, y = AXIS == 0 ? j : i;
      if (i <= 2) {
        const double edge = j == 0 ? 2.0 * PI * pw[i + 1] : PI * pw[i + 1] * (oma * (1.0 + a));
        G.m[x][y] = fma(cc, m, G.m[x][y]);
        G.e[x][y] = fma(cc, fma(q + 1.0, m, edge), G.e[x][y]);
      }
      if (q >= 1) G.g[x][y] = fma(cc, m + hh, G.g[x][y]);
    }
}

// Full disk: the moments of the unit sphere, 4pi (1), 4pi/3 (w1^2), 4pi/15
// (w1^2 w2^2); zero for odd powers; hhat = m / q.
__device__ __forceinline__ void add_full(Moments& G, double c) {
  const double m0 = 4.0 * PI * c, m2 = 4.0 * PI / 3.0 * c, m22 = 4.0 * PI / 15.0 * c;
  G.m[0][0] += m0;
  G.e[0][0] += m0;
  G.m[2][0] += m2;
  G.m[0][2] += m2;
  G.e[2][0] += 3.0 * m2;
  G.e[0][2] += 3.0 * m2;
  G.g[2][0] += 1.5 * m2;
  G.g[0][2] += 1.5 * m2;
  G.m[2][2] += m22;
  G.e[2][2] += 5.0 * m22;
  G.g[2][2] += 1.25 * m22;
}

// tanh-sinh rule on [0, 1]: nodes x = 1/(1 + e^{-2u}), u = (pi/2) sinh(t), t = k/16.
// The integrands are bounded at x = 0 and grow as (1 - x)^{-1/2} at x = 1, so
// nodes below k = -55 (weights under 1e-20) and above 64 add nothing.
constexpr int RULE_FIRST = -55, RULE_NODES = 120;
struct Rule {
  double x[RULE_NODES], omx[RULE_NODES], w[RULE_NODES];
};
__device__ __forceinline__ void fill_rule(Rule& R, int n) {
  const double t = (n + RULE_FIRST) * (1.0 / 16.0);
  const double u = 0.5 * PI * sinh(t), cu = cosh(u);
  R.w[n] = 0.5 * (1.0 / 16.0) * 0.5 * PI * cosh(t) / (cu * cu);
  R.x[n] = 1.0 / (1.0 + exp(-2.0 * u));
  R.omx[n] = 1.0 / (1.0 + exp(2.0 * u));
}

// Double cap {xi >= a, eta >= b}, a, b >= 0, by the lanes of an aligned group of
// four (`lane` 0..3), each of which receives the whole result.
__device__ __forceinline__ void double_cap(const Rule& R, int lane, double a, double b,
                                           Moments& M) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (i < 3 && j < 3) M.m[i][j] = M.e[i][j] = 0.0;
      M.g[i][j] = 0.0;
    }
  const double a2 = a * a, b2 = b * b, pb2 = a2 + b2;
  if (!(pb2 < 1.0)) return;  // (the same in all four lanes)
  const double pb = sqrt(pb2), L = (1.0 - pb2) / (1.0 + pb);
  // p - a and p - b from their values at p = pb (no cancellation there)
  const double pa0 = pb > 0.0 ? b2 / (pb + a) : 0.0, pb0 = pb > 0.0 ? a2 / (pb + b) : 0.0;
  const double a3 = a2 * a, b3 = b2 * b;
#pragma unroll 1
  for (int n = lane; n < RULE_NODES; n += 4) {
    const double Lx = L * R.x[n], omp = L * R.omx[n], p = pb + Lx;
    const double rs = rsqrt(omp * (1.0 + p)), sq = omp * (1.0 + p) * rs;
    const double wl = 2.0 * L * R.w[n];
    const double W1 = wl * p * rs, W = fma(wl, sq / p, W1);  // weights of m, of m + hhat
    const double u2 = (pa0 + Lx) * (p + a), v2 = (pb0 + Lx) * (p + b);
    const double u = sqrt(u2), v = sqrt(v2), p2 = p * p;
    // arc moments between (v, b) and (a, u) on the circle of radius p
    const double B00 = atan2(fmax(fma(u, v, -a * b), 0.0), fma(a, v, u * b));
    const double B10 = u - b, B01 = v - a, B11 = 0.5 * (u2 - b2);
    const double xy = fma(a, u, -v * b), pB = p2 * B00;
    const double B20 = 0.5 * (pB + xy), B02 = 0.5 * (pB - xy);
    const double x2y = fma(a2, u, -v2 * b), xy2 = fma(a, u2, -v * b2);
    const double t3 = 1.0 / 3.0, p10 = p2 * B10, p01 = p2 * B01;
    const double B30 = t3 * fma(2.0, p10, x2y), B21 = t3 * (p01 + xy2),
                 B12 = t3 * (p10 - x2y), B03 = t3 * fma(2.0, p01, -xy2);
    const double x3y = fma(a3, u, -(v2 * v) * b), x2y2 = fma(a2, u2, -v2 * b2);
    const double p11 = 2.0 * p2 * B11;
    const double B31 = 0.25 * (p11 + x2y2), B13 = 0.25 * (p11 - x2y2),
                 B22 = 0.25 * fma(p2, B20, -x3y);
    M.m[0][0] = fma(W1, B00, M.m[0][0]);
    M.m[1][0] = fma(W1, B10, M.m[1][0]);
    M.m[0][1] = fma(W1, B01, M.m[0][1]);
    M.m[2][0] = fma(W1, B20, M.m[2][0]);
    M.m[1][1] = fma(W1, B11, M.m[1][1]);
    M.m[0][2] = fma(W1, B02, M.m[0][2]);
    M.m[2][1] = fma(W1, B21, M.m[2][1]);
    M.m[1][2] = fma(W1, B12, M.m[1][2]);
    M.m[2][2] = fma(W1, B22, M.m[2][2]);
    M.g[1][0] = fma(W, B10, M.g[1][0]);
    M.g[0][1] = fma(W, B01, M.g[0][1]);
    M.g[2][0] = fma(W, B20, M.g[2][0]);
    M.g[1][1] = fma(W, B11, M.g[1][1]);
    M.g[0][2] = fma(W, B02, M.g[0][2]);
    M.g[3][0] = fma(W, B30, M.g[3][0]);
    M.g[2][1] = fma(W, B21, M.g[2][1]);
    M.g[1][2] = fma(W, B12, M.g[1][2]);
    M.g[0][3] = fma(W, B03, M.g[0][3]);
    M.g[3][1] = fma(W, B31, M.g[3][1]);
    M.g[2][2] = fma(W, B22, M.g[2][2]);
    M.g[1][3] = fma(W, B13, M.g[1][3]);
  }
  const unsigned four = 0xfu << (threadIdx.x & 28u);
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (i < 3 && j < 3) M.m[i][j] += __shfl_xor_sync(four, M.m[i][j], o);
        if (has_g(i, j)) M.g[i][j] += __shfl_xor_sync(four, M.g[i][j], o);
      }
  }
  // r d/dr m(a = dx/r, b = dy/r) = -a dm/da - b dm/db; the derivatives are minus
  // the line integrals of xi^i eta^j Psi along xi = a and eta = b
  const double sa = sqrt((1.0 - a) * (1.0 + a)), sb = sqrt((1.0 - b) * (1.0 + b));
  const double sp = sqrt((1.0 - pb) * (1.0 + pb));
  const double xa = fmin(b / sa, 1.0), ca = fmin(sp / sa, 1.0);  // sine, cosine of the line's end
  const double xb = fmin(a / sb, 1.0), cb = fmin(sp / sb, 1.0);
  const double pha = acos(xa), phb = acos(xb);
  const double Ia[3] = {pha, ca, 0.5 * fma(xa, ca, pha)}, Ib[3] = {phb, cb, 0.5 * fma(xb, cb, phb)};
  const double sa_[3] = {1.0, sa, sa * sa}, sb_[3] = {1.0, sb, sb * sb};
  const double a_[3] = {a, a2, a3}, b_[3] = {b, b2, b3};  // a a^i, b b^j
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      M.e[i][j] = fma(i + j + 1.0, M.m[i][j],
                      2.0 * fma(a_[i], sa_[j] * Ia[j], b_[j] * (sb_[i] * Ib[i])));
}

// Moments of the region {xi >= lam, eta >= mu} (V) for any signs; D is the double
// cap at (|lam|, |mu|).
__device__ __forceinline__ void region_xy(double lam, double mu, const Moments& D, Moments& G) {
  const bool nx = lam < 0.0, ny = mu < 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // (-1)^(nx + ny) times the double cap reflected in the negative axes
      const bool neg = ((nx ? i + 1 : 0) + (ny ? j + 1 : 0)) & 1;
      if (i < 3 && j < 3) {
        G.m[i][j] = neg ? -D.m[i][j] : D.m[i][j];
        G.e[i][j] = neg ? -D.e[i][j] : D.e[i][j];
      }
      G.g[i][j] = neg ? -D.g[i][j] : D.g[i][j];
    }
  if (ny) add_single<0>(G, nx ? -1.0 : 1.0, fabs(lam), nx);
  if (nx) add_single<1>(G, ny ? -1.0 : 1.0, fabs(mu), ny);
  if (nx && ny) add_full(G, 1.0);
}

// Moments of {xi >= lam} (AXIS 0) or {eta >= lam} (AXIS 1) for any sign.
template <int AXIS>
__device__ __forceinline__ void region_half(double lam, Moments& G) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (i < 3 && j < 3) G.m[i][j] = G.e[i][j] = 0.0;
      G.g[i][j] = 0.0;
    }
  if (lam < 0.0) add_full(G, 1.0);
  add_single<AXIS>(G, lam < 0.0 ? -1.0 : 1.0, fabs(lam), lam < 0.0);
}

// Coefficients (1, X, X^2) of the Q2 Lagrange basis l_0, l_1, l_2 at local
// coordinate s = sF + 2X (X the offset from F in units of h).
__device__ __forceinline__ void basis_about(double sF, double B[3][3]) {
  B[0][0] = 0.5 * sF * (sF - 1.0); B[0][1] = 2.0 * sF - 1.0; B[0][2] = 2.0;
  B[1][0] = 1.0 - sF * sF;         B[1][1] = -4.0 * sF;      B[1][2] = -4.0;
  B[2][0] = 0.5 * sF * (sF + 1.0); B[2][1] = 2.0 * sF + 1.0; B[2][2] = 2.0;
}

// nodal values f[ix][iy] -> monomial coefficients about F, axis by axis
__device__ __forceinline__ void monomials(const double f[3][3], const double Bx[3][3],
                                          const double By[3][3], double P[3][3]) {
  double t[3][3];
#pragma unroll
  for (int ix = 0; ix < 3; ++ix)
#pragma unroll
    for (int q = 0; q < 3; ++q)
      t[ix][q] = fma(f[ix][0], By[0][q], fma(f[ix][1], By[1][q], f[ix][2] * By[2][q]));
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int q = 0; q < 3; ++q)
      P[p][q] = fma(t[0][q], Bx[0][p], fma(t[1][q], Bx[1][p], t[2][q] * Bx[2][p]));
}

// One fragment's (pi, u, v) * 4pi; P, U, V are its (pi, u, v) deviations in
// monomials about F.
__device__ __forceinline__ void contract(const Moments& M, const double P[3][3],
                                         const double U[3][3], const double V[3][3], double r,
                                         double acc[3]) {
  double rq[5];
  rq[0] = 1.0;
#pragma unroll
  for (int k = 1; k < 5; ++k) rq[k] = rq[k - 1] * r;
  acc[0] = acc[1] = acc[2] = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      double t0 = P[a][b] * M.e[a][b], t1 = 0.0, t2 = 0.0;
      if (a > 0) {
        t0 = fma(-a * U[a][b], M.m[a - 1][b], t0);
        t1 = a * (fma(U[a][b], M.g[a][b], V[a][b] * M.g[a - 1][b + 1]) -
                  P[a][b] * M.m[a - 1][b]);
      }
      if (b > 0) {
        t0 = fma(-b * V[a][b], M.m[a][b - 1], t0);
        t2 = b * (fma(V[a][b], M.g[a][b], U[a][b] * M.g[a + 1][b - 1]) -
                  P[a][b] * M.m[a][b - 1]);
      }
      acc[0] = fma(rq[a + b], t0, acc[0]);
      acc[1] = fma(rq[a + b], t1, acc[1]);
      acc[2] = fma(rq[a + b], t2, acc[2]);
    }
}

}  // namespace fc

constexpr int FC_THREADS = 128;

// Foot-centred point update of family FAM (0 V, 1 E_v, 2 E_h), FP64: a group of
// NF lanes (one per adjacent cell) per point and duration; writes the half-step
// and new point planes.  `t`: the thread's index over all lanes of the family.
template <int FAM>
__device__ __forceinline__ void point_fc(const StepArgs<double>& a, const fc::Rule& R, size_t t) {
  using namespace fc;
  constexpr int NF = FAM == 0 ? 4 : 2;
  const int k = (int)(t % NF), s = (int)(t / NF) & 1;
  const size_t id = t / (2 * NF);
  if (id >= (size_t)a.nx * a.ny) return;  // (whole groups leave together)
  const int j = (int)(id / a.nx), i = (int)(id - (size_t)j * a.nx);
  LatticeG<double> L = lattice_of(a);
  const int I = 2 * i + (FAM == 2 ? 1 : 0);
  const int J = 2 * j + (FAM == 1 ? 1 : 0);
  const Prim<double> wp = L.at(I, J);
  unsigned bad = 0;
  // the lane's cell: its side of the lines x = x_P and y = y_P
  const double sx = FAM == 2 ? 1.0 : ((FAM == 0 ? (k == 1 || k == 2) : k == 1) ? -1.0 : 1.0);
  const double sy = FAM == 1 ? 1.0 : ((FAM == 0 ? k >= 2 : k == 1) ? -1.0 : 1.0);
  const double th = (s == 0 ? 0.5 * a.dt : a.dt) * (1.0 / a.h);
  // two-Picard convective foot (Eq. adv-footpoint), then the frozen state at F
  const double d1x = -th * wp.u, d1y = -th * wp.v;
  const Prim<double> w1 = eval_w(L, locate<double>(I, J, d1x, d1y));
  const double fx = -th * w1.u, fy = -th * w1.v;  // F - P, units of h
  const Prim<double> ws = eval_w(L, locate<double>(I, J, fx, fy));
  if (!(ws.r > 0.0 && ws.p > 0.0)) bad |= FLAG_NONPHYSICAL;
  const double cs = sqrt(a.gas.gamma * ws.p / ws.r), Z = ws.r * cs, Zi = 1.0 / Z;
  const double r = cs * th;
  if (!(fabs(fx) + r < 0.5 && fabs(fy) + r < 0.5)) bad |= FLAG_CFL | FLAG_REACH;
  const double rr = fmax(r, 1e-300);
  // everything below is in the frame reflected by (sx, sy): the cell's nodes lie at
  // P + (ix, iy) half cells (edge families: centred on P along the edge)
  const double rx = sx * fx, ry = sy * fy;
  const double lam = -rx / rr, mu = -ry / rr;  // the lines through P, scaled
  Moments G;
  if constexpr (FAM == 0) {
    Moments D;
    double_cap(R, k, fabs(lam), fabs(mu), D);
    region_xy(lam, mu, D, G);
  } else if constexpr (FAM == 1) {
    region_half<0>(lam, G);
  } else {
    region_half<1>(mu, G);
  }
  // the cell's Q2 data as deviations from W_*, in monomials about F
  double Bx[3][3], By[3][3];
  basis_about((FAM == 2 ? 0.0 : -1.0) + 2.0 * rx, Bx);
  basis_about((FAM == 1 ? 0.0 : -1.0) + 2.0 * ry, By);
  double fp[3][3], fu[3][3], fv[3][3], P[3][3], U[3][3], V[3][3];
  const int isx = sx > 0.0 ? 1 : -1, isy = sy > 0.0 ? 1 : -1;
#pragma unroll
  for (int ix = 0; ix < 3; ++ix)
#pragma unroll
    for (int iy = 0; iy < 3; ++iy) {
      const Prim<double> w = L.at(FAM == 2 ? I - 1 + ix : I + isx * ix,
                                  FAM == 1 ? J - 1 + iy : J + isy * iy);
      fp[ix][iy] = (w.p - ws.p) * Zi;
      fu[ix][iy] = sx * (w.u - ws.u);
      fv[ix][iy] = sy * (w.v - ws.v);
    }
  monomials(fp, Bx, By, P);
  monomials(fu, Bx, By, U);
  monomials(fv, Bx, By, V);
  double acc[3];
  contract(G, P, U, V, rr, acc);
  // the cell holding F gives the data value at F (the last one where several do)
  const bool holds = (FAM == 2 || rx >= 0.0) && (FAM == 1 || ry >= 0.0);
  const unsigned group = ((NF == 4 ? 0xfu : 0x3u) << (threadIdx.x & 31u & ~(NF - 1u)));
  const unsigned have = __ballot_sync(group, holds) & group;
  const int src = have ? 31 - __clz(have) : (int)(threadIdx.x & 31u & ~(NF - 1u));
  const double u0 = have ? __shfl_sync(group, sx * U[0][0], src) : 0.0;
  const double v0 = have ? __shfl_sync(group, sy * V[0][0], src) : 0.0;
  acc[1] *= sx;
  acc[2] *= sy;
#pragma unroll
  for (int o = 1; o < NF; o <<= 1)
#pragma unroll
    for (int q = 0; q < 3; ++q) acc[q] += __shfl_xor_sync(group, acc[q], o);
  if (k != 0) return;
  Prim<double> nw;
  const double k4 = 1.0 / (4.0 * PI);
  nw.p = ws.p + Z * (acc[0] * k4);
  nw.u = ws.u + (u0 + acc[1] * k4);
  nw.v = ws.v + (v0 + acc[2] * k4);
  nw.r = ws.r + (nw.p - ws.p) / (cs * cs);
  if (!(isfinite(nw.r) && isfinite(nw.u) && isfinite(nw.v) && isfinite(nw.p)))
    bad |= FLAG_NONFINITE;
  double* const* dst = s == 0 ? a.half[FAM] : a.out.pt[FAM];
  dst[0][id] = nw.r;
  dst[1][id] = nw.u;
  dst[2][id] = nw.v;
  dst[3][id] = nw.p;
  raise_flag(a.flags, bad);
}

// All three families in one launch: blocks [0, nv) take the vertices (eight lanes
// per point), then E_v and E_h with ne blocks each (four lanes per point).
__global__ void __launch_bounds__(FC_THREADS) k_points_fc(StepArgs<double> a, int nv, int ne) {
  __shared__ fc::Rule R;
  const int b = blockIdx.x;
  if (b < nv) {
    if (threadIdx.x < fc::RULE_NODES) fc::fill_rule(R, threadIdx.x);
    __syncthreads();
    point_fc<0>(a, R, (size_t)b * FC_THREADS + threadIdx.x);
  } else if (b < nv + ne) {
    point_fc<1>(a, R, (size_t)(b - nv) * FC_THREADS + threadIdx.x);
  } else {
    point_fc<2>(a, R, (size_t)(b - nv - ne) * FC_THREADS + threadIdx.x);
  }
}

}  // namespace af
