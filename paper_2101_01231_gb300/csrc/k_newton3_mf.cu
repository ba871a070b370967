// Matrix-free Newton prediction of 3D Burgers at degree 1 (Sec. 2.2, Sec. 3), one CTA per region,
// ahead of the dense per-region LU of k_newton3.cu (which solves the regions left over).
//
// At degree 1 the residual's rule has two Gauss points per dimension, at which phi_1 = +-1: the
// node values of a cell are sums and differences of its modes, and the residual and its exact
// Jacobian (for Burgers the quasi-quadrature-free one) act on them pointwise, by 2 x 2 matrices
// along lines and through face traces.  A thread holds one column (cell, z, y, x) of the 27
// cells with its two time nodes in registers; the derivative partner comes by shuffle, only
// the values for the face traces go through shared memory.  The linear systems are solved by
// BiCGStab in FP32 with the time operator as preconditioner, as in k_newton_mf.cuh; the FP64
// form refines each one against its FP64 residual down to round-off, so that the iterates are
// the dense LU's.
//
// The dense LU costs 54 MFLOP per region and iteration and moves its trailing matrix through
// L2 for each of 432 columns; here a region takes ~0.1 M FP64 operations per iteration, and
// the FP64 pipe and the barriers of the ~10 applications per solve bound it.  Measured, one
// step of 10 x 11 x 9 cells in FP64 (with the nodal correction of k_newton3.cu): 585 -> 0.97 ms,
// of it 0.83 ms this kernel (2.35 ms before the FP32 copies were kept from being reconverted).
#include <cuda_runtime.h>

#include "k_nl_lines.cuh"
#include "nl3.h"
#include "ridg_internal.h"

namespace ridg {
namespace {

constexpr int kCols = 216, kNT = 224, kNW = kNT / 32;
constexpr int kFaceLines = 432;  // 3 directions x 9 rows x 4 faces x 4 tangential nodes
constexpr int kMaxRefine3 = 8, kMaxInner3 = 32;
constexpr double kS3 = 1.7320508075688772935;

// the two face lines of a thread: first nodes left / right of the face (-1 outside the
// region), the node stride along the normal
struct Lines3 {
  int bl[2], br[2], st[2];
};

// the linearisation point: the column's values, the traces of its face lines, alpha / 2
template <typename T>
struct Lin3 {
  T w[2], wl[2][2], wr[2][2], al[2];
};

// the column's constants: lam D, +-lam E of its node per direction, its face values' places
template <typename T>
struct Col3 {
  T kd[3], pd[3], md[3];
  int fl[3];
};

// traces of P (node values [t][column]) on the thread's face line k
template <typename T>
__device__ __forceinline__ void line_traces(const T* P, const Lines3& L, int k, int t, T& l, T& r) {
  const T lo = T(0.5 * (1.0 - kS3)), hi = T(0.5 * (1.0 + kS3));
  const T* p = P + t * kCols;
  l = L.bl[k] >= 0 ? lo * p[L.bl[k]] + hi * p[L.bl[k] + L.st[k]] : T(0);
  r = L.br[k] >= 0 ? hi * p[L.br[k]] + lo * p[L.br[k] + L.st[k]] : T(0);
}

// Surface minus volume terms on node values.  LINEAR: of J v at the linearisation S; else of
// the residual at v.  P: [t][column], Fh: [t][face line].  (Two barriers; the caller
// synchronises before the next call.)
template <typename T, bool LINEAR>
__device__ __forceinline__ void spatial(const Col3<T>& C, const Lines3& L, const Lin3<T>& S,
                                        const T (&v)[2], T (&out)[2], T* P, T* Fh) {
  const int tid = threadIdx.x;
  T g[2];
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    g[t] = LINEAR ? S.w[t] * v[t] : T(0.5) * v[t] * v[t];
    if (tid < kCols) P[t * kCols + tid] = v[t];
  }
  __syncthreads();
  if (tid < kCols) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        T l, r;
        line_traces(P, L, k, t, l, r);
        const T fl = LINEAR ? S.wl[k][t] * l : T(0.5) * l * l;
        const T fr = LINEAR ? S.wr[k][t] * r : T(0.5) * r * r;
        Fh[t * kFaceLines + tid + k * kCols] =
            L.bl[k] < 0 ? fr : L.br[k] < 0 ? fl : T(0.5) * (fl + fr) - S.al[k] * (r - l);
      }
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    T acc = T(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T gs = g[t] + __shfl_xor_sync(0xffffffffu, g[t], 1 << d);
      const T* f = Fh + t * kFaceLines + C.fl[d];
      acc += C.kd[d] * gs + C.pd[d] * f[4] + C.md[d] * f[0];
    }
    out[t] = acc;
  }
}

// node values to modes (and back, unnormalised): butterflies over z, y, x of a cell's lanes,
// time in registers
__device__ __forceinline__ void to_modes(double (&v)[2]) {
#pragma unroll
  for (int b = 1; b < 8; b <<= 1)
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const double o = __shfl_xor_sync(0xffffffffu, v[t], b);
      v[t] = 0.5 * ((threadIdx.x & b) ? v[t] - o : v[t] + o);
    }
  const double a = v[0];
  v[0] = 0.5 * (a + v[1]);
  v[1] = 0.5 * (v[1] - a);
}

template <bool F64>
__global__ void __launch_bounds__(kNT, 4) newton3_mf_kernel(const Newton3Args a) {
  __shared__ double Pd[2 * kCols], Fd[2 * kFaceLines], alpha[108];
  __shared__ float red[8 * kNW];
  float* P = (float*)Pd;
  float* Fh = (float*)Fd;
  const int tid = threadIdx.x;
  const bool col = tid < kCols;
  const int r = col ? tid >> 3 : 0, node = tid & 7;
  const long long e = blockIdx.x;
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  const int c3[3] = {r % 3, (r / 3) % 3, r / 9};
  // node values of the column's Q, extended constant in time
  double w[2], q = 0.0;
  {
    const unsigned u = (unsigned)e, uz = u / (unsigned)(nx * ny), ur = u - uz * (unsigned)(nx * ny);
    int cx = (int)(ur % (unsigned)nx) + c3[0] - 1, cy = (int)(ur / (unsigned)nx) + c3[1] - 1,
        cz = (int)uz + c3[2] - 1;
    cx += cx < 0 ? nx : (cx >= nx ? -nx : 0);
    cy += cy < 0 ? ny : (cy >= ny ? -ny : 0);
    cz += cz < 0 ? nz : (cz >= nz ? -nz : 0);
    q = a.Q[(((long long)cz * ny + cy) * nx + cx) * 8 + node];
#pragma unroll
    for (int b = 1; b < 8; b <<= 1) {
      const double o = __shfl_xor_sync(0xffffffffu, q, b);
      q = (node & b) ? o + q : q - o;  // phi_1 = -1 at the lower node
    }
    if (!col) q = 0.0;
  }
  w[0] = w[1] = q;
  Lines3 L;
  Col3<double> C;
  Col3<float> Cf;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int i = (col ? tid : 0) + k * kCols, f = i >> 2, o = i & 3, d = f / 36,
              row = (f - 36 * d) >> 2, pos = f & 3;
    const int cell = d == 0 ? 3 * row : d == 1 ? row % 3 + 9 * (row / 3) : row;
    const int cs = d == 0 ? 1 : d == 1 ? 3 : 9;
    const int nb = d == 0 ? 2 * o : d == 1 ? (o & 1) + 4 * (o >> 1) : o;
    L.st[k] = 1 << d;
    L.bl[k] = pos > 0 ? (cell + (pos - 1) * cs) * 8 + nb : -1;
    L.br[k] = pos < 3 ? (cell + pos * cs) * 8 + nb : -1;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const bool up = node >> d & 1;
    C.kd[d] = up ? -a.lam[d] * kS3 : a.lam[d] * kS3;
    C.pd[d] = a.lam[d] * (up ? 1.0 + kS3 : 1.0 - kS3);
    C.md[d] = -a.lam[d] * (up ? 1.0 - kS3 : 1.0 + kS3);
    const float lf = nl::keep((float)a.lam[d]), sf = (float)kS3;
    Cf.kd[d] = up ? -lf * sf : lf * sf;
    Cf.pd[d] = lf * (up ? 1.f + sf : 1.f - sf);
    Cf.md[d] = -lf * (up ? 1.f - sf : 1.f + sf);
    const int row = d == 0 ? c3[1] + 3 * c3[2] : d == 1 ? c3[0] + 3 * c3[2] : c3[0] + 3 * c3[1];
    const int o = d == 0 ? node >> 1 : d == 1 ? (node & 1) + 2 * (node >> 2) : node & 3;
    C.fl[d] = Cf.fl[d] = (d * 36 + row * 4 + c3[d]) * 4 + o;
  }
  int buf = 0, it = 0;
  float m1[1] = {(float)fabs(q)};
  nl::reduce<kNW, 1, true>(m1, red, buf);
  double wnorm = m1[0];  // the iterate's largest entry (below FP32's range by its high word)
  if (wnorm < 1e-30) {
    nl::MaxAbs m;
    m.add(q);
    wnorm = __hiloint2double(nl::block_max_hi<kNW>(m, red, buf), 0);
  }
  // Rusanov speeds of the initial iterate: the largest trace of both sides over the face
  if (col) Pd[tid] = q;
  if (tid < 108) alpha[tid] = 0.0;
  __syncthreads();
  Lin3<double> S;
  if (col)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      double l, rr;
      line_traces(Pd, L, k, 0, l, rr);
      // (non-negative doubles order like their bits)
      if (L.bl[k] >= 0 && L.br[k] >= 0)
        atomicMax((unsigned long long*)&alpha[(tid + k * kCols) >> 2],
                  (unsigned long long)__double_as_longlong(fmax(fabs(l), fabs(rr))));
    }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 2; ++k) S.al[k] = col ? 0.5 * alpha[(tid + k * kCols) >> 2] : 0.0;
  // time operator on node values ([[1, s], [-s, 3]] on modes, s = sqrt 3), its inverse
  const double T00 = 2.0, T01 = kS3 - 1.0, T10 = -1.0 - kS3, T11 = 2.0;
  const double det = T00 * T11 - T01 * T10;
  const float I00 = (float)(T11 / det), I01 = (float)(-T01 / det), I10 = (float)(-T10 / det),
              I11 = (float)(T00 / det);
  bool conv = false, capped = false;
#pragma unroll 1
  for (; it < a.max_iters;) {
    // FP64 residual; psi_a(-1) summed over the time modes is 1 + s and 1 - s at the nodes
    double R[2], x[2];
    spatial<double, false>(C, L, S, w, R, Pd, Fd);
    R[0] += T00 * w[0] + T01 * w[1] - (1.0 + kS3) * q;
    R[1] += T10 * w[0] + T11 * w[1] - (1.0 - kS3) * q;
    // linearisation (P still holds w)
    Lin3<float> Sf;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      S.w[t] = w[t];
      Sf.w[t] = nl::keep((float)w[t]);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        line_traces(Pd, L, k, t, S.wl[k][t], S.wr[k][t]);
        Sf.wl[k][t] = nl::keep((float)S.wl[k][t]);
        Sf.wr[k][t] = nl::keep((float)S.wr[k][t]);
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) Sf.al[k] = nl::keep((float)S.al[k]);
    __syncthreads();
    ++it;
    bool ok = true;
    x[0] = x[1] = 0.0;
#pragma unroll 1
    for (int ref = 0;; ++ref) {
      nl::MaxAbs rm;
      if (col) {
        rm.add(R[0]);
        rm.add(R[1]);
      }
      const int rhi = nl::block_max_hi<kNW>(rm, red, buf);
      ok = rhi < nl::kHi1e30 && ref < kMaxRefine3;
      if (!ok) break;
      const int ex = nl::exponent_of(rhi);
      const double scale = nl::pow2(-ex), unscale = nl::pow2(ex);
      const float wrel = (float)(wnorm * scale);  // wnorm on the right-hand side's scale
      // BiCGStab
      float rv[2], rh[2], p[2], v[2], t[2], xf[2] = {0.f, 0.f};
      {
        const float b0 = nl::keep((float)(R[0] * scale)), b1 = nl::keep((float)(R[1] * scale));
        rv[0] = col ? I00 * b0 + I01 * b1 : 0.f;
        rv[1] = col ? I10 * b0 + I11 * b1 : 0.f;
      }
      rh[0] = p[0] = rv[0];
      rh[1] = p[1] = rv[1];
      m1[0] = rv[0] * rv[0] + rv[1] * rv[1];
      nl::reduce<kNW, 1, false>(m1, red, buf);
      const float bb = m1[0], bmean = sqrtf(bb / (2 * kCols));
      const float tol = fminf(F64 ? 1e-3f : 1e-2f, fmaxf(F64 ? 3e-6f : 1e-6f, (F64 ? 1e-17f : 1e-15f) * wrel / bmean));
      const float stop = tol * tol * bb;
      float rho = bb, rr = bb, hh = bb;
      auto apply = [&](const float (&in)[2], float (&out)[2]) {
        float s[2];
        spatial<float, true>(Cf, L, Sf, in, s, P, Fh);
        out[0] = in[0] + I00 * s[0] + I01 * s[1];
        out[1] = in[1] + I10 * s[0] + I11 * s[1];
        if (!col) out[0] = out[1] = 0.f;
      };
#pragma unroll 1
      for (int k = 0; k < 2 * kMaxInner3 && rr > stop; ++k) {
        if (k == kMaxInner3) {  // stalled: again with another shadow vector (k_newton_mf.cuh)
          if (rr <= 0.1f * bb) break;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            p[i] = rv[i];
            rh[i] = (tid & 1) ? 0.f : rv[i];
          }
          m1[0] = rh[0] * rv[0] + rh[1] * rv[1];
          nl::reduce<kNW, 1, false>(m1, red, buf);
          rho = hh = m1[0];
        }
        apply(p, v);
        m1[0] = rh[0] * v[0] + rh[1] * v[1];
        nl::reduce<kNW, 1, false>(m1, red, buf);
        const float al = rho / m1[0];
        rv[0] -= al * v[0];
        rv[1] -= al * v[1];
        apply(rv, t);
        float s4[4] = {t[0] * rv[0] + t[1] * rv[1], t[0] * t[0] + t[1] * t[1],
                       rh[0] * t[0] + rh[1] * t[1], rv[0] * rv[0] + rv[1] * rv[1]};
        nl::reduce<kNW, 4, false>(s4, red, buf);
        const float om = s4[1] > 0.f ? s4[0] / s4[1] : 0.f;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          xf[i] += al * p[i] + om * rv[i];
          rv[i] -= om * t[i];
        }
        rr = fmaxf(0.f, s4[3] - om * s4[0]);
        if (!(fabsf(al) < 1e30f) || !(rr < 1e30f)) {
          ok = false;
          break;
        }
        const float rho1 = -om * s4[2];
        if (rho1 * rho1 <= 1e-5f * rr * hh) {  // about to stall: start anew (k_newton_mf.cuh)
          rh[0] = p[0] = rv[0];
          rh[1] = p[1] = rv[1];
          rho = hh = rr;
          continue;
        }
        const float be = rho1 / rho * (al / om);
        rho = rho1;
#pragma unroll
        for (int i = 0; i < 2; ++i) p[i] = rv[i] + be * (p[i] - om * v[i]);
      }
      if (!ok || rr > 0.1f * bb) {
        ok = false;
        break;
      }
      const float ratio = bb > 0.f ? sqrtf(rr / bb) : 0.f;
      double z[2] = {unscale * (double)xf[0], unscale * (double)xf[1]};
      x[0] += z[0];
      x[1] += z[1];
      if (!F64) break;
      m1[0] = fmaxf(fabsf(xf[0]), fabsf(xf[1]));
      nl::reduce<kNW, 1, true>(m1, red, buf);
      // what is left of the linear system is below the iterate's round-off
      if (m1[0] * fmaxf(ratio, 1e-6f) <= 5e-17f * wrel) break;
      double Jz[2];
      spatial<double, true>(C, L, S, z, Jz, Pd, Fd);
      R[0] -= Jz[0] + T00 * z[0] + T01 * z[1];
      R[1] -= Jz[1] + T10 * z[0] + T11 * z[1];
      __syncthreads();
    }
    if (!ok) break;
    double dm[2] = {x[0], x[1]}, wm[2];
    w[0] -= x[0];
    w[1] -= x[1];
    wm[0] = w[0];
    wm[1] = w[1];
    to_modes(dm);
    to_modes(wm);
    float mx[2] = {0.f, 0.f};
    if (col) {
      mx[0] = isfinite(dm[0]) && isfinite(dm[1])
                  ? __double2float_ru(fmax(fabs(dm[0]), fabs(dm[1]))) : 3e38f;
      mx[1] = isfinite(wm[0]) && isfinite(wm[1])
                  ? __double2float_rd(fmax(fabs(wm[0]), fabs(wm[1]))) : 3e38f;
    }
    nl::reduce<kNW, 2, true>(mx, red, buf);
    if (!(mx[0] < 1e30f) || !(mx[1] < 1e30f)) break;
    wnorm = mx[1];
    if (wnorm < 1e-30) {
      nl::MaxAbs m;
      if (col) {
        m.add(wm[0]);
        m.add(wm[1]);
      }
      wnorm = __hiloint2double(nl::block_max_hi<kNW>(m, red, buf), 0);
    }
    if ((double)mx[0] <= a.tol * fmax(1.0, (double)mx[1])) {
      conv = true;
    } else {
      // the FP64 iterates are the dense LU's to round-off, also at the cap (one region sent there
      // costs 32 ms; a tolerance below round-off, where the two differ, stays its to decide)
      capped = F64 && it == a.max_iters && (double)mx[0] > 1e-12 * fmax(1.0, (double)mx[1]);
    }
    if (conv || capped) {
      if (col && r == 13) {
        a.W[e * 16 + node] = wm[0];
        a.W[e * 16 + 8 + node] = wm[1];
      }
      break;
    }
  }
  if (tid == 0) {
    if (conv || capped) {
      if (!conv) atomicAdd(&a.stats[0], 1);
      atomicMax(&a.stats[1], it);
      atomicAdd(&a.stats[7 + (it < 15 ? it : 15)], 1);
      atomicAdd(a.iters_total, (unsigned long long)it);
    } else {
      a.list[atomicAdd(a.list_count, 1)] = (int)e;
    }
  }
}

}  // namespace

cudaError_t launch_newton3_mf(bool fp32, const Newton3Args& a, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(a.list_count, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  if (fp32)
    newton3_mf_kernel<false><<<(unsigned)a.ncell, kNT, 0, s>>>(a);
  else
    newton3_mf_kernel<true><<<(unsigned)a.ncell, kNT, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace ridg
