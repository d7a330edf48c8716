// af_reduce.cuh -- FP64 global diagnostics of a state: conserved totals
// (Sec. 3.1), the entropy functional -int rho log(p/rho^gamma) dA (Sec. 6),
// kinetic energy, wave-speed / positivity extrema and the vorticity integral
// (Sec. 6.4).  Two passes: per-block partials with warp shuffles, then one
// block folds the partials in a fixed order (bitwise reproducible).
//
// What bounds them: the FP64 unit (two lanes per cycle and SM).  A cell took about
// 575 of its instructions: ten CUDA logarithms, eight square roots and seven
// divisions, 32 conversions, minima and maxima.  It takes 170 now: the
// logarithm by a table (8 instructions, below), conversions on the integer units,
// the minima on the stored floats, the wave speed evaluated in FP64 only where its
// FP32 value comes near the grid's largest one, which the centre recovery before it
// finds; common factors taken out of the sums.
// A call at 2048^2 in FP32_COMP: 1.52 ms, 4.69 before (of which 0.22 ms was the
// fold of the partials by one thread per value, now one warp); the FP64 unit is 82%
// busy in k_inv_partial.  (1.34 ms with a logarithm whose leading part was rounded and
// with storage offsets added in plain FP32, which missed the largest speed beside a
// dense reference.)
#pragma once

#include "af_common.cuh"
#include "af_log_table.cuh"
#include "af_ref_kernels.cuh"

namespace af {

enum { RED_SUMS = 8, RED_VALS = 11, RED_THREADS = 128, RED_WARPS = RED_THREADS / 32 };
// partial layout: sums mass, mx, my, E, 9 x entropy(Simpson), entropy(avg), KE,
// 6/h x vorticity; then max(|u|+c), min rho, min p

template <typename T>
struct RedArgs {
  Planes<T> st;
  const T* wc[4];
  int nx, ny;
  double gamma, h;
  double rho_ref, p_ref, e_ref;  // storage offsets (see Gas)
  TopSpeed top;         // the grid's largest FP32 wave speed (k_center found it)
  double* partial;      // [RED_VALS][gridDim.x]
};

// ---- logarithm by table (P. T. P. Tang, "Table-driven implementation of the
// logarithm function in IEEE floating-point arithmetic", ACM TOMS 16, 1990) ----
// x = 2^e m with m in [0.707, 1.414); c the nearest of 512 points (nine bits of m), g
// near 1/c, r = g m - 1 (|r| < 2^-9.8): log x = e log 2 - log g + log(1 + r), the last by
// its series.  The leading part e log 2 - log g is exact (both terms are multiples of
// 2^-42, what they leave is a float, gen_log_table.py); the terms from r^4 on, below 2^-31
// of r, and the sum of the left-over parts are FP32; everything else is FP64.  At the point
// next to 1, which is 1 itself, log g = 0 and small results keep their relative
// accuracy.  Error 1.03 ulp at most (where the sum crosses a power of two next to 1) and
// 0.27 rms; CUDA's log has 0.54 and 0.25; with the leading part rounded it was 1.8 and
// 0.44.  The entropies, sums of 3200 cells, are within 2.1 (nodes) and 3.0 (averages)
// units of 2^-53 rms of extended precision; with CUDA's log they were within 2.5 and 3.1.
struct LogTable {
  LogEntry e[LOG_POINTS];
  float lo[LOG_POINTS];
};
__device__ __forceinline__ void fill_log_table(LogTable& tab, int thread, int threads) {
  for (int i = thread; i < LOG_POINTS; i += threads) {
    tab.e[i] = LOG_TABLE[i];
    tab.lo[i] = LOG_TABLE_LO[i];
  }
}
__device__ __forceinline__ double log_by_table(double x, const LogTable& tab) {
  const unsigned hi = (unsigned)__double2hiint(x);
  if (hi - 0x00100000u >= 0x7fe00000u) return log(x);  // not a positive normal number
  const unsigned t = hi - LOG_FIRST + 0x400u;  // (+ half a point: the nearest one)
  const int e = (int)t >> 20, i = (int)((t & 0xfffffu) >> 11);
  const LogEntry c = tab.e[i];
  const double m = __hiloint2double((int)(hi - ((unsigned)e << 20)), __double2loint(x));
  const double r = fma(m, c.g, -1.0);
  const float ef = (float)e, rf = narrow(r);
  const double head = fma(widen(ef), LOG_2_HI, c.hi);  // exact
  const float lo = fmaf(ef, LOG_2_LO, tab.lo[i]);
  const float tail = fmaf(rf, fmaf(rf, -1.0f / 6.0f, 0.2f), -0.25f);
  const double q = fma(r, fma(r, widen(tail), 1.0 / 3.0), -0.5);
  return head + (r + fma(r * r, q, widen(lo)));
}

__device__ __forceinline__ double entropy_density(double r, double p, double gamma,
                                                  const LogTable& tab) {
  return r * fma(gamma, log_by_table(r, tab), -log_by_table(p, tab));
}

// running minimum of stored values (NaN ignored)
__device__ __forceinline__ void keep_min(float& m, float x) { m = fminf(m, x); }
__device__ __forceinline__ void keep_min(double& m, double x) {
  // signed-integer order of the bits (sign-magnitude turned into two's complement)
  const long long a = __double_as_longlong(x), b = __double_as_longlong(m);
  const bool nan = (a & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
  const long long ka = a < 0 ? a ^ 0x7fffffffffffffffll : a;
  const long long kb = b < 0 ? b ^ 0x7fffffffffffffffll : b;
  if (!nan && ka < kb) m = x;
}

__device__ __forceinline__ double wide(float x) { return widen(x); }
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ bool same_bits(float x, float y) {
  return __float_as_uint(x) == __float_as_uint(y);
}
__device__ __forceinline__ bool same_bits(double x, double y) {
  return __double_as_longlong(x) == __double_as_longlong(y);
}

// |u| + c of a node (absolute rho, p)
__device__ __forceinline__ double wave_speed(double r, double u, double v, double p,
                                             double gamma) {
  return sqrt(fma(u, u, v * v)) + sqrt(gamma * p / r);
}

template <typename T, bool COMP>
__global__ void __launch_bounds__(RED_THREADS) k_inv_partial(const __grid_constant__ RedArgs<T> a) {
  __shared__ LogTable tab;
  __shared__ double sh[RED_WARPS][RED_VALS];
  fill_log_table(tab, threadIdx.x, RED_THREADS);
  __syncthreads();
  double acc[RED_SUMS] = {};
  double smax = 0.0;
  const float near_top = __uint_as_float(*a.top.bits) * (1.f - 1e-6f);
  T seen[4] = {};          // (rho, u, v, p) of the lane's last FP64 wave speed,
  bool any_seen = false;   // if it has taken one
  T rmin = (T)INFINITY, pmin = (T)INFINITY;  // of the stored offsets
  const size_t N = (size_t)a.nx * a.ny;
  for (size_t id = (size_t)blockIdx.x * RED_THREADS + threadIdx.x; id < N;
       id += (size_t)gridDim.x * RED_THREADS) {
    const int j = (int)(id / (unsigned)a.nx), i = (int)(id - (size_t)j * a.nx);
    const int ip = i + 1 == a.nx ? 0 : i + 1, jp = j + 1 == a.ny ? 0 : j + 1;
    // every load of the cell first
    const T* const* const pl[4] = {a.st.pt[0], a.st.pt[1], a.st.pt[2], a.wc};
    T w[4][4], av[4], lo[4];
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int k = 0; k < 4; ++k) w[n][k] = pl[n][k][id];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      av[k] = a.st.avg[k][id];
      if (COMP) lo[k] = a.st.lo[k][id];
    }
    const size_t q10 = (size_t)j * a.nx + ip, q01 = (size_t)jp * a.nx + i,
                 q11 = (size_t)jp * a.nx + ip;
    const T v10 = a.st.pt[0][2][q10], u10 = a.st.pt[0][1][q10];
    const T v11 = a.st.pt[0][2][q11], u11 = a.st.pt[0][1][q11];
    const T v01 = a.st.pt[0][2][q01], u01 = a.st.pt[0][1][q01];
    const T vev10 = a.st.pt[1][2][q10], ueh01 = a.st.pt[2][1][q01];
    // averages
    double ub[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ub[k] = wide(av[k]);
      if (COMP) ub[k] += wide(lo[k]);
      if (sizeof(T) == 4 && k == 0) ub[k] += a.rho_ref;
      if (sizeof(T) == 4 && k == 3) ub[k] += a.e_ref;
      acc[k] += ub[k];
    }
    const double ke = 0.5 * fma(ub[1], ub[1], ub[2] * ub[2]) / ub[0];
    acc[5] += entropy_density(ub[0], (a.gamma - 1.0) * (ub[3] - ke), a.gamma, tab);
    acc[6] += ke;
    // The Simpson entropy integral sums, over the cells, the nine nodes of each
    // with weights (1/6, 4/6, 1/6) x (1/6, 4/6, 1/6).  On the periodic grid every
    // vertex lies in four cells, every edge midpoint in two and every centre in
    // one, so the same total is each cell's own four nodes (vertex (i, j), edges
    // (i, j+1/2) and (i+1/2, j), centre) with weights 1/9, 2/9, 2/9, 4/9.
    double H[4];
    float sf[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const double r = sizeof(T) == 4 ? wide(w[n][0]) + a.rho_ref : wide(w[n][0]);
      const double p = sizeof(T) == 4 ? wide(w[n][3]) + a.p_ref : wide(w[n][3]);
      H[n] = entropy_density(r, p, a.gamma, tab);
      keep_min(rmin, w[n][0]);
      keep_min(pmin, w[n][3]);
      sf[n] = wave_speed_f32(a.top.rho_ref, a.top.p_ref, w[n][0], w[n][1], w[n][2], w[n][3],
                             a.top.gamma);
    }
    // The wave speed in FP64 only at nodes whose FP32 value is within 1e-6 of the
    // grid's largest.  k_center found that one by the same operations on the same
    // stored values, so the node that gave it is always among them; each FP32 value is
    // within 3e-7 of its node's, so the node of the largest FP64 value is too.
#pragma unroll 1
    for (int n = 0; n < 4; ++n) {
      const float sn = n == 0 ? sf[0] : n == 1 ? sf[1] : n == 2 ? sf[2] : sf[3];
      if (!(sn >= near_top)) continue;
      T q[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        q[k] = n == 0 ? w[0][k] : n == 1 ? w[1][k] : n == 2 ? w[2][k] : w[3][k];
      if (any_seen && same_bits(q[0], seen[0]) && same_bits(q[1], seen[1]) &&
          same_bits(q[2], seen[2]) && same_bits(q[3], seen[3]))
        continue;
      any_seen = true;
#pragma unroll
      for (int k = 0; k < 4; ++k) seen[k] = q[k];
      const double rr = sizeof(T) == 4 ? wide(q[0]) + a.rho_ref : wide(q[0]);
      const double pp = sizeof(T) == 4 ? wide(q[3]) + a.p_ref : wide(q[3]);
      smax = fmax(smax, wave_speed(rr, wide(q[1]), wide(q[2]), pp, a.gamma));
    }
    acc[4] += fma(4.0, H[3], fma(2.0, H[1] + H[2], H[0]));
    // circulation around the cell: Simpson along its four edges (the right and
    // top edges' nodes belong to the neighbouring cells), differences first
    const double cv = fma(4.0, wide(vev10) - wide(w[1][2]),
                          (wide(v10) - wide(w[0][2])) + (wide(v11) - wide(v01)));
    const double cu = fma(4.0, wide(ueh01) - wide(w[2][1]),
                          (wide(u01) - wide(w[0][1])) + (wide(u11) - wide(u10)));
    acc[7] += cv - cu;
  }
  // block reduction: warp shuffles, then the warp results in order
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double off = sizeof(T) == 4 ? 1.0 : 0.0;
  double vals[RED_VALS];
#pragma unroll
  for (int k = 0; k < RED_SUMS; ++k) vals[k] = acc[k];
  vals[8] = smax;
  vals[9] = wide(rmin) + off * a.rho_ref;
  vals[10] = wide(pmin) + off * a.p_ref;
#pragma unroll
  for (int k = 0; k < RED_VALS; ++k) {
    double v = vals[k];
    for (int o = 16; o > 0; o >>= 1) {
      double t = __shfl_down_sync(0xffffffffu, v, o);
      v = (k < RED_SUMS) ? v + t : (k == 8 ? fmax(v, t) : fmin(v, t));
    }
    if (lane == 0) sh[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < RED_VALS) {
    int k = threadIdx.x;
    double v = sh[0][k];
    for (int wi = 1; wi < RED_WARPS; ++wi)
      v = (k < RED_SUMS) ? v + sh[wi][k] : (k == 8 ? fmax(v, sh[wi][k]) : fmin(v, sh[wi][k]));
    a.partial[(size_t)k * gridDim.x + blockIdx.x] = v;
  }
}

// One block of RED_VALS warps: warp k folds value k of the nblocks partials, each
// lane its share in index order, then the lanes by shuffles; `out` is the host's
// pinned memory, written through the device's mapping.
__global__ void k_inv_final(const double* partial, int nblocks, double h, double* out,
                            unsigned* top) {
  if (threadIdx.x == 0) *top = 0u;  // for the next call
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* pk = partial + (size_t)k * nblocks;
  // (one branch per warp: selecting among sum, max and min inside the loop would
  // issue all three on the FP64 unit, 20 us instead of 5)
  auto fold = [&](double v, auto op) {
#pragma unroll 8
    for (int b = lane; b < nblocks; b += 32) v = op(v, pk[b]);
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
  };
  double v;
  if (k < RED_SUMS)
    v = fold(0.0, [](double x, double y) { return x + y; });
  else if (k == 8)
    v = fold(0.0, [](double x, double y) { return fmax(x, y); });
  else
    v = fold(INFINITY, [](double x, double y) { return fmin(x, y); });
  if (lane != 0) return;
  // output order follows AF_INV_*: mass, mx, my, E, entropy, entropy_avg, KE,
  // max speed, min rho, min p, vorticity
  const double h2 = h * h;
  if (k < 7) out[k] = (k == 4 ? h2 / 9.0 : h2) * v;
  else if (k == 7) out[10] = h / 6.0 * v;
  else out[k - 1] = v;
  __threadfence_system();
}

}  // namespace af
