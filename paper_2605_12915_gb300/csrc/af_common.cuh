// af_common.cuh -- device building blocks shared by the kernels of the RB-TAI
// Active Flux step: gas model (Sec. 2), Q2 Lagrange basis (Sec. 4), the
// half-cell lattice addressing of the point values, error bits.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace af {

// device error bits (latched with atomicOr; mapped to af_status on the host)
enum : unsigned {
  FLAG_CFL = 1u,          // c_K dt / h > 1/2 at a node
  FLAG_NONPHYSICAL = 2u,  // rho <= 0 or p <= 0 where c is needed
  FLAG_NONFINITE = 4u,    // NaN / Inf in the new state
  FLAG_REACH = 8u,        // convective foot more than one cell from its point
  FLAG_TIMEOUT = 16u,     // a bounded wait for the CTA's own asynchronous copies ran out
  FLAG_BOUNDS = 32u       // debug builds (AF_BOUNDS_CHECK): a checked index left its region
};

template <typename T>
struct Prim {
  T r, u, v, p;
};

template <typename T>
struct PUV {
  T p, u, v;
};

// raw pointers to the sixteen planes of a state (and the four lo planes of the
// compensated averages; null unless AF_FP32_COMP)
template <typename T>
struct Planes {
  T* avg[4];
  T* pt[3][4];  // [family V, E_v, E_h][rho, u, v, p]
  T* lo[4];
};

__device__ __forceinline__ int wrapi(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

// ---- gas model (Sec. 2) ---------------------------------------------------
// Storage convention: density and pressure are held as offsets from a
// per-grid reference state (rho_ref, p_ref), and the energy average as an
// offset from p_ref/(gamma-1).  In FP32 this keeps the rounding of stored
// values proportional to the flow's variations rather than to the absolute
// pressure (low-Mach flows carry p ~ 1/(gamma M^2)); in FP64 the offsets are 0.
template <typename T>
struct Gas {
  T gamma, gm1, gm1inv, g_gm1;  // gamma, gamma-1, 1/(gamma-1), gamma/(gamma-1)
  T rho_ref, p_ref;
};

// The absolute value of a stored offset.  In FP64 the offsets' reference is 0 and
// the value is the stored one (no addition).
__device__ __forceinline__ float with_ref(float ref, float x) { return ref + x; }
__device__ __forceinline__ double with_ref(double, double x) { return x; }

// Tests on the bits of a double: a comparison is an instruction of the FP64 unit,
// which takes 64 cycles for a warp here (two lanes per cycle and SM), an integer
// one takes one or two.  Same answers as the comparisons, NaN included (at_least_one
// alone takes a positive NaN for a number: its caller has sorted NaN out).
__device__ __forceinline__ bool is_positive(float x) { return x > 0.f; }
__device__ __forceinline__ bool is_positive(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool is_finite(float x) { return isfinite(x); }
__device__ __forceinline__ bool is_finite(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}
// |x| > lim for a positive finite lim (false for NaN)
__device__ __forceinline__ bool abs_above(float x, float lim) { return fabsf(x) > lim; }
__device__ __forceinline__ bool abs_above(double x, double lim) {
  const long long b = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return b > __double_as_longlong(lim) && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool is_negative(float x) { return x < 0.f; }
__device__ __forceinline__ bool is_negative(double x) {
  const long long b = __double_as_longlong(x);
  return b < 0 && b != (long long)0x8000000000000000ull;
}
__device__ __forceinline__ bool at_least_one(float x) { return x >= 1.f; }
__device__ __forceinline__ bool at_least_one(double x) { return __double2hiint(x) >= 0x3ff00000; }

// (float)x and (double)x on the integer units (the conversion instructions run at
// the FP64 unit's rate): the exponent is rebiased and the mantissa shifted, with
// round to nearest even on narrowing.  Same values as the instructions, subnormals,
// infinities and NaN included; none of the branches holds an FP64 instruction, which
// would be issued, predicated off, for every warp.
__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned a = hi & 0x7fffffffu, sign = hi & 0x80000000u;
  if (a - 0x38100000u < 0x0fe00000u) {  // exponents of normal floats
    unsigned m = __funnelshift_l(lo, a - 0x38000000u, 3);
    m += ((lo << 3) + (m & 1u)) > 0x80000000u ? 1u : 0u;
    return __uint_as_float(m | sign);
  }
  if (a >= 0x47f00000u)  // beyond the floats: infinity, or NaN
    return __uint_as_float(a > 0x7ff00000u || (a == 0x7ff00000u && lo) ? 0x7fffffffu
                                                                      : sign | 0x7f800000u);
  // below 2^-126: round(|x| 2^149), the bits of a subnormal float
  const unsigned e = a >> 20, sh = 926u - e;
  if (sh > 63u) return __uint_as_float(sign);
  const unsigned long long M =
      ((unsigned long long)((a & 0xfffffu) | 0x100000u) << 32) | lo;
  unsigned long long q = M >> sh;
  const unsigned long long rest = M << (64u - sh), half = 1ull << 63;
  if (rest > half || (rest == half && (q & 1ull))) ++q;
  return __uint_as_float(sign | (unsigned)q);
}
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), a = u & 0x7fffffffu, sign = u & 0x80000000u;
  unsigned hi = (a >> 3) + 0x38000000u, lo = u << 29;
  if (a - 0x00800000u >= 0x7f000000u) {
    if (a >= 0x7f800000u) {  // infinity, NaN
      hi = 0x7ff00000u | ((a & 0x7fffffu) >> 3);
    } else {  // zero, or a subnormal: a 2^-149 by way of the float a
      const unsigned b = __float_as_uint(__uint2float_rn(a));
      hi = a ? (b >> 3) + 0x38000000u - (149u << 20) : 0u;
      lo = b << 29;
    }
  }
  return __hiloint2double((int)(sign | hi), (int)lo);
}

// Programmatic dependent launch: the next kernel of the stream may be scheduled
// now (its blocks then sit in pdl_wait), and this one's input is complete.  A
// kernel launched without the attribute passes both at once.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The helpers below spell out their fused multiply-adds: the library is built
// without contraction, so every copy of an expression rounds the same way (a
// value computed by two thread blocks must agree bitwise for conservation).

// conservative offsets (rho~, rho u, rho v, E~) of a stored primitive
// (rho~, u, v, p~): E~ = E - p_ref/(gamma-1) = p~/(gamma-1) + rho |u|^2 / 2
template <typename T>
__device__ __forceinline__ void cons_from_stored(const Prim<T>& w, const Gas<T>& g, T u[4]) {
  const T rho = with_ref(g.rho_ref, w.r);
  u[0] = w.r;
  u[1] = rho * w.u;
  u[2] = rho * w.v;
  u[3] = fma(w.p, g.gm1inv, (T(0.5) * rho) * fma(w.u, w.u, w.v * w.v));
}

// primitive from conservative offsets given 1/rho
template <typename T>
__device__ __forceinline__ Prim<T> stored_from_cons_inv(const T u[4], const Gas<T>& g, T inv) {
  Prim<T> w;
  w.r = u[0];
  w.u = u[1] * inv;
  w.v = u[2] * inv;
  w.p = g.gm1 * fma(T(-0.5), fma(u[1], w.u, u[2] * w.v), u[3]);
  return w;
}

template <typename T>
__device__ __forceinline__ Prim<T> stored_from_cons(const T u[4], const Gas<T>& g) {
  return stored_from_cons_inv(u, g, T(1) / with_ref(g.rho_ref, u[0]));
}

// Euler fluxes F (x) and G (y) of a stored primitive.  The constant p_ref is
// left out of the momentum fluxes: it cancels in every flux difference.
template <typename T>
__device__ __forceinline__ void flux_x(const Prim<T>& w, const Gas<T>& g, T f[4]) {
  const T rho = with_ref(g.rho_ref, w.r), p = with_ref(g.p_ref, w.p);
  const T m = rho * w.u;
  f[0] = m;
  f[1] = fma(m, w.u, w.p);
  f[2] = m * w.v;
  f[3] = w.u * fma(p, g.g_gm1, (T(0.5) * rho) * fma(w.u, w.u, w.v * w.v));
}

template <typename T>
__device__ __forceinline__ void flux_y(const Prim<T>& w, const Gas<T>& g, T f[4]) {
  const T rho = with_ref(g.rho_ref, w.r), p = with_ref(g.p_ref, w.p);
  const T m = rho * w.v;
  f[0] = m;
  f[1] = m * w.u;
  f[2] = fma(m, w.v, w.p);
  f[3] = w.v * fma(p, g.g_gm1, (T(0.5) * rho) * fma(w.u, w.u, w.v * w.v));
}

__device__ __forceinline__ float narrow_any(float x) { return x; }
__device__ __forceinline__ float narrow_any(double x) { return narrow(x); }

// A storage offset's reference as the sum of two floats (hi nearest, lo the rest)
struct RefPair {
  float hi, lo;
};
// The absolute value (hi + lo) + x to 2^-24 of itself (and 2^-49 of the reference), also
// where hi and x cancel, as they do at a light node beside a dense reference: the
// rounding of hi + x is recovered exactly.
__device__ __forceinline__ float with_ref_pair(RefPair ref, float x) {
  const float s = ref.hi + x, b = s - ref.hi;
  return s + (((ref.hi - (s - b)) + (x - b)) + ref.lo);
}
__device__ __forceinline__ float with_ref_pair(RefPair, double x) { return narrow(x); }

// |u| + c of a stored node in FP32, within 5 x 2^-24 = 3e-7 relative.  Roundings, in
// units of 2^-24: c^2 five (gamma, rho, p, quotient, product), which the root halves
// and adds one to; |u| four (1.5 of the quotient t, whose square enters with weight 1/2 at
// most, 0.5 of the sum under the root, the root, the larger component); the final sum
// one.  Infinity where FP32 cannot tell: an overflow, an underflow, an infinity or NaN
// in any of the values.
template <typename T>
__device__ __forceinline__ float wave_speed_f32(RefPair rho_ref, RefPair p_ref, T r_, T u_, T v_,
                                                T p_, float gamma) {
  const float r = with_ref_pair(rho_ref, r_), p = with_ref_pair(p_ref, p_);
  const float u = narrow_any(u_), v = narrow_any(v_);
  const float a = fmaxf(fabsf(u), fabsf(v)), b = fminf(fabsf(u), fabsf(v));
  const float t = a > 0.f ? b / a : 0.f;
  const float c2 = gamma * (p / r);
  if (!(c2 > 1e-30f) || !(fminf(r, p) > 1e-37f) || (a > 0.f && a < 1e-30f)) return INFINITY;
  // (the last term is 0, or NaN if u or v is NaN or infinite: maxima and minima drop NaN)
  const float s = fmaf(a, sqrtf(fmaf(t, t, 1.f)), sqrtf(c2)) + 0.f * (u + v);
  return s < INFINITY ? s : INFINITY;
}

// ---- Q2 Lagrange basis on nodes -1, 0, 1 (Sec. 4) ----------------------------
template <typename T>
__device__ __forceinline__ void lagrange3(T s, T l[3]) {
  T hs = T(0.5) * s;
  l[0] = hs * (s - T(1));
  l[1] = T(1) - s * s;
  l[2] = hs * (s + T(1));
}

// ---- half-cell lattice ------------------------------------------------------
// Every point of the Q2 reconstruction lives on the lattice of half cells:
// lattice (I, J) = (2i + a, 2j + b) is, for (a, b) = (0,0) the vertex V(i,j),
// (0,1) the x-edge midpoint E_v(i,j), (1,0) the y-edge midpoint E_h(i,j) and
// (1,1) the centre of C_ij.  Cell C_ij owns lattice nodes 2i..2i+2 x 2j..2j+2.
__device__ __forceinline__ int lattice_family(int I, int J) {
  return (I & 1) ? ((J & 1) ? 3 : 2) : ((J & 1) ? 1 : 0);
}

// Global-memory view of the lattice: the point planes of one state plus the
// recovered centres (family 3).
template <typename T>
struct LatticeG {
  const T* f[4][4];  // [family][rho, u, v, p]
  int nx, ny;
  __device__ __forceinline__ Prim<T> at(int I, int J) const {
    int fam = lattice_family(I, J);
    int i = wrapi(I >> 1, nx), j = wrapi(J >> 1, ny);
    size_t id = (size_t)j * nx + i;
    Prim<T> w;
    w.r = f[fam][0][id];
    w.u = f[fam][1][id];
    w.v = f[fam][2][id];
    w.p = f[fam][3][id];
    return w;
  }
};

// ---- error-free transformations (compensated averages) ---------------------
// Knuth's TwoSum: s + e == a + b exactly (round-to-nearest, no contraction).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Compensated average update: (hi, lo) <- (hi, lo) + (fl - fr) + (gb - gt),
// with fl, fr, gb, gt the scaled edge terms shared with the neighbouring cells.
// Every step before the last is error free (Knuth TwoSum), so each edge value
// enters its two cells with opposite signs exactly and the only rounding is
// that of the new lo word.
__device__ __forceinline__ void comp_update(float& hi, float& lo, float fl, float fr, float gb,
                                            float gt) {
  float dx, ex, dy, ey, d, ed, s, es, t, et;
  two_sum(fl, -fr, dx, ex);
  two_sum(gb, -gt, dy, ey);
  two_sum(dx, dy, d, ed);
  two_sum(hi, d, s, es);
  two_sum(lo, es, t, et);
  t = __fadd_rn(t, __fadd_rn(et, __fadd_rn(ed, __fadd_rn(ex, ey))));
  hi = __fadd_rn(s, t);
  lo = __fsub_rn(t, __fsub_rn(hi, s));
}

}  // namespace af
