// FP64 building blocks of the 2D nonlinear path's sum-factorised quadrature: transforms of one
// line of modes or Gauss-point values held in registers, and the physical fluxes of a point.
//
// The FP64 pipe (2 FMA per clock and SM) bounds every kernel that uses them, so they spend
// registers to save FP64 operations: the Gauss points are symmetric and phi_b is even or odd,
// so the values at x_q and -x_q share their even and odd partial sums (NB = 3 modes to 4
// points: 6 FMA instead of 12; 5 to 7: 20 instead of 35).
#pragma once

#include <cuda_runtime.h>

#include "k_nlflux.cuh"

namespace ridg {
namespace nl {

// The residual's points per dimension, ceil((3M + 1) / 2).
constexpr int residual_points(int nb) { return (3 * (nb - 1) + 2) / 2; }

// An NP-point Gauss rule for NB modes.  Its lower half is kept, q < H, with the centre point
// at H - 1 if NP is odd.
template <int NB, int NP = residual_points(NB)>
struct Rule {
  static constexpr int NQ = NP, H = (NQ + 1) / 2;
  double V[NB][H];     // phi_b(x_q)
  double wV[NB][H];    // w_q phi_b(x_q)
  double wD[NB][H];    // w_q phi_b'(x_q)
  double ep[NB];       // phi_b(+1); phi_b(-1) = (-1)^b phi_b(+1)
};
// host (k_newton_mf.cu): NB = 2 .. 5 with NP = residual_points(NB) or 2 NB - 1
template <int NB, int NP = residual_points(NB)>
Rule<NB, NP> make_rule();

// the traces at +1 (e + o) and -1 (e - o) of the polynomial with modes m[0], m[st], ...
template <int NB, int NQ>
__device__ __forceinline__ void traces(const Rule<NB, NQ>& T, const double* m, int st, double& e,
                                       double& o) {
  e = m[0];
  o = T.ep[1] * m[st];
#pragma unroll
  for (int b = 2; b < NB; ++b)
    if (b & 1) o = fma(T.ep[b], m[b * st], o); else e = fma(T.ep[b], m[b * st], e);
}

// values at the NQ points of the polynomial with modes a
template <int NB, int NQ>
__device__ __forceinline__ void interp(const Rule<NB, NQ>& T, const double (&a)[NB],
                                       double (&v)[NQ]) {
#pragma unroll
  for (int q = 0; q < NQ / 2; ++q) {
    double e = a[0];
#pragma unroll
    for (int b = 2; b < NB; b += 2) e = fma(T.V[b][q], a[b], e);
    if constexpr (NB <= 3) {
      v[q] = fma(T.V[1][q], a[1], e);
      v[NQ - 1 - q] = fma(-T.V[1][q], a[1], e);
    } else {
      const double o = fma(T.V[3][q], a[3], T.V[1][q] * a[1]);
      v[q] = e + o;
      v[NQ - 1 - q] = e - o;
    }
  }
  if constexpr (NQ & 1) {
    double e = a[0];
#pragma unroll
    for (int b = 2; b < NB; b += 2) e = fma(T.V[b][NQ / 2], a[b], e);
    v[NQ / 2] = e;
  }
}

// out[b] = sum_q w_q phi_b(x_q) f[q], or with phi_b'
template <bool DERIV, int NB, int NQ>
__device__ __forceinline__ void project(const Rule<NB, NQ>& T, const double (&f)[NQ],
                                        double (&out)[NB]) {
  constexpr int HP = NQ / 2;
  double s[HP], d[HP];
#pragma unroll
  for (int q = 0; q < HP; ++q) {
    s[q] = f[q] + f[NQ - 1 - q];
    d[q] = f[q] - f[NQ - 1 - q];
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if constexpr (DERIV) {
      if (b == 0) {
        out[b] = 0.0;
        continue;
      }
    }
    const bool even = DERIV ? (b & 1) : !(b & 1);
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < HP; ++q) {
      const double w = DERIV ? T.wD[b][q] : T.wV[b][q];
      const double x = even ? s[q] : d[q];
      acc = q == 0 ? w * x : fma(w, x, acc);
    }
    if constexpr (NQ & 1)
      if (even) acc = fma(DERIV ? T.wD[b][HP] : T.wV[b][HP], f[HP], acc);
    out[b] = acc;
  }
}

// phi_b(x_q), and w_q phi_b(x_q), at any q (compile-time indices)
template <int NB, int NQ>
__device__ __forceinline__ double vq(const Rule<NB, NQ>& T, int b, int q) {
  constexpr int H = (NQ + 1) / 2;
  return q < H ? T.V[b][q] : ((b & 1) ? -T.V[b][NQ - 1 - q] : T.V[b][NQ - 1 - q]);
}
template <int NB, int NQ>
__device__ __forceinline__ double wvq(const Rule<NB, NQ>& T, int b, int q) {
  constexpr int H = (NQ + 1) / 2;
  return q < H ? T.wV[b][q] : ((b & 1) ? -T.wV[b][NQ - 1 - q] : T.wV[b][NQ - 1 - q]);
}

// 1 / x by Newton-Raphson, r += r (1 - x r), two steps from the hardware's approximation (relative
// error 2^-20): 2^-80 ahead of the last rounding, so the correctly rounded value but where 1 / x
// lies that close to the middle of two (one x in some 10^8, and x = 1 - 2^-53), there its
// neighbour.  Four FP64 operations, where the division takes about three times as many on the
// same pipe (Euler Q2, 160^2, a step 12.6 ms; with __drcp_rn 12.9).  For 2^-1022 <= |x| <= 2^1022:
// 0, subnormal and non-finite x give NaN, larger finite ones 0.  The solver refuses such a density
// (a NaN, or an iterate above 1e30), and its region is block-eliminated, with divisions.
__device__ __forceinline__ double reciprocal(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// u = w1 / rho, v = w2 / rho.  ANY: also for densities outside the reciprocal's range, by divisions
// (the correction, whose states go to no other solver).
template <bool ANY>
__device__ __forceinline__ void velocity(const double* w, double& u, double& v) {
  const double ir = reciprocal(w[0]);
  u = w[1] * ir;
  v = w[2] * ir;
  if constexpr (ANY) {
    const unsigned hi = (unsigned)__double2hiint(w[0]) & 0x7fffffffu;
    if (hi - 0x00100000u >= 0x7fd00000u - 0x00100000u) {
      u = w[1] / w[0];
      v = w[2] / w[0];
    }
  }
}

// both directions' fluxes of one state (Euler: one reciprocal), or one's
template <int FLUX, bool ANY = false>
__device__ __forceinline__ void flux2(const double* w, double* fx, double* fy, double g) {
  if constexpr (FLUX == RIDG_FLUX_BURGERS) {
    fx[0] = 0.5 * w[0] * w[0];
  } else {
    double u, v;
    velocity<ANY>(w, u, v);
    const double p = (g - 1.0) * (w[3] - 0.5 * fma(w[1], u, w[2] * v)), h = w[3] + p;
    fx[0] = w[1];
    fx[1] = fma(w[1], u, p);
    fx[2] = w[1] * v;
    fx[3] = u * h;
    fy[0] = w[2];
    fy[1] = fx[2];
    fy[2] = fma(w[2], v, p);
    fy[3] = v * h;
  }
}
template <int FLUX, bool ANY = false>
__device__ __forceinline__ void flux1(const double* w, int dd, double* f, double g) {
  if constexpr (FLUX == RIDG_FLUX_BURGERS) {
    f[0] = 0.5 * w[0] * w[0];
  } else {
    double u, v;
    velocity<ANY>(w, u, v);
    const double p = (g - 1.0) * (w[3] - 0.5 * fma(w[1], u, w[2] * v));
    const double un = dd == 0 ? u : v;
    f[0] = dd == 0 ? w[1] : w[2];
    f[1] = w[1] * un;
    f[2] = w[2] * un;
    if (dd == 0) f[1] += p; else f[2] += p;
    f[3] = un * (w[3] + p);
  }
}

// F'(w) z of both directions, or of one (Euler: of the state's primitives)
template <int FLUX>
__device__ __forceinline__ void dflux2(const double* w, const double* z, double* fx, double* fy,
                                       double g) {
  if constexpr (FLUX == RIDG_FLUX_BURGERS) {
    fx[0] = w[0] * z[0];
  } else {
    const double ir = reciprocal(w[0]), u = w[1] * ir, v = w[2] * ir, k = 0.5 * fma(u, u, v * v);
    const double H = (w[3] + (g - 1.0) * fma(-w[0], k, w[3])) * ir;
    const double dp = (g - 1.0) * (fma(k, z[0], z[3]) - fma(u, z[1], v * z[2]));
    const double a = fma(-u, z[0], z[1]), b = fma(-v, z[0], z[2]), h = z[3] + dp;
    fx[0] = z[1];
    fx[1] = fma(u, z[1] + a, dp);
    fx[2] = fma(v, a, u * z[2]);
    fx[3] = fma(H, a, u * h);
    fy[0] = z[2];
    fy[1] = fma(u, b, v * z[1]);
    fy[2] = fma(v, z[2] + b, dp);
    fy[3] = fma(H, b, v * h);
  }
}
template <int FLUX>
__device__ __forceinline__ void dflux1(const double* w, const double* z, int dd, double* f,
                                       double g) {
  if constexpr (FLUX == RIDG_FLUX_BURGERS) {
    f[0] = w[0] * z[0];
  } else {
    double fx[4], fy[4];
    dflux2<FLUX>(w, z, fx, fy, g);
#pragma unroll
    for (int j = 0; j < 4; ++j) f[j] = dd ? fy[j] : fx[j];
  }
}

// An FP32 value made from FP64 ones that is kept, not recomputed: where registers run short the
// compiler otherwise repeats the conversion (an FP64-pipe instruction) at every use.
__device__ __forceinline__ float keep(float x) {
  asm volatile("" : "+f"(x));
  return x;
}

// Block reduction of NV sums (or maxima) over NW warps, one barrier; red holds 8 NW floats, and
// buf alternates between calls so that the next one needs no barrier before it.
template <int NW, int NV, bool MAX>
__device__ __forceinline__ void reduce(float (&v)[NV], float* red, int& buf) {
  static_assert(NV <= 4, "four slots per warp");
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float t = __shfl_xor_sync(0xffffffffu, v[k], o);
      v[k] = MAX ? fmaxf(v[k], t) : v[k] + t;
    }
  float* p = red + buf * 4 * NW;
  buf ^= 1;
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) p[(threadIdx.x >> 5) * 4 + k] = v[k];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    v[k] = p[k];
#pragma unroll
    for (int w = 1; w < NW; ++w) v[k] = MAX ? fmaxf(v[k], p[w * 4 + k]) : v[k] + p[w * 4 + k];
  }
}

// The largest |x| of a thread's FP64 values by their high words (positive doubles order like
// their bits; no FP64 operation): a lower bound to 2^-20, infinite if one is not finite.
struct MaxAbs {
  int hi = 0;
  __device__ __forceinline__ void add(double x) { hi = max(hi, __double2hiint(x) & 0x7fffffff); }
};

// the block's largest high word (as FP32 patterns, which order like integers up to 0x7f7fffff;
// larger ones, |x| >= 2^1008 or not finite, are cut)
template <int NW>
__device__ __forceinline__ int block_max_hi(MaxAbs m, float* red, int& buf) {
  float v[1] = {__int_as_float(min(m.hi, 0x7f000000))};
  reduce<NW, 1, true>(v, red, buf);
  return __float_as_int(v[0]);
}
constexpr int kHi1e30 = 0x46293e59;  // high word of 1e30

// The exponent of a right-hand side whose largest high word is hi, within the normal range, and
// the power of two of one: right-hand sides are scaled to a maximum of 1 to 2 before they become
// FP32, whatever the state's scale.
__device__ __forceinline__ int exponent_of(int hi) { return max((hi >> 20) - 1023, -1022); }
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

}  // namespace nl
}  // namespace ridg
