// Matrix-free Newton prediction for a nonlinear flux in 2D (Sec. 3): the first solver of every
// precision, one CTA per region.
//
// The region system of eq. pred_full_system is solved by the same outer iteration as in
// k_newton.cuh -- FP64 residual by quadrature, FP64 iterate, stop when ||dW||_inf <=
// tol max(1, ||W||_inf); the mixed precisions solve the linear systems in FP32, the FP64 form
// refines those solutions against the linear system's FP64 residual down to round-off -- but
// no Jacobian is stored and nothing is factorised:
//  * the linearised residual is applied in FP32 on the nodal basis of the NB^3 Gauss points
//    of every cell, where a product with F'(w) is pointwise and a derivative is one NB x NB
//    matrix per line (the integrals int d Psi_k Psi_l F'(w) by NB points per dimension);
//  * the time operator (psi_a(1) psi_g(1) - int psi_a' psi_g, one NB x NB matrix) is the
//    preconditioner.  The step is an integral equation in time, so the preconditioned operator
//    is a small perturbation of the identity at the scheme's time steps and BiCGStab reaches
//    1e-4 .. 1e-5 in 3 to 12 iterations (two applications each).
// A direct solve needs 118 b^3 flop per region and factorisation (b = m theta_T unknowns per
// cell: 149 MFLOP for Euler Q2) and moves every block through L2; one application here is
// ~30 kFMA for Euler Q2 and its data stay in shared memory and registers.  What bounds the
// kernel is the FP64 pipe (2 FMA per clock and SM), on the two or three FP64 residuals that
// the outer iteration cannot do without; those are evaluated by sum factorisation along lines
// held in registers, with the even / odd symmetry of the Gauss points (about half the
// multiplications), one flux evaluation per point for both directions and one per face.
// Measured against the block elimination alone (one step with its correction, tensor-core /
// FP32 solves): Euler Q2 160^2 214 -> 12.6 ms (the residuals' FP64 operations alone: 8.8 ms),
// Euler Q1 67 x 90 7.7 -> 0.91 ms, eight Burgers problems of up to 72^2 at degrees 1 .. 4
// 227 -> 9.7 ms; FP64, Burgers Q2 45 x 33 31.7 -> 0.55 ms.
//
// The initial iterate is Q^n extended constant in time, so the first residual is evaluated
// with one time mode and one time point.
//
// A region that does not converge quickly (mixed: contraction below 10x per solve; BiCGStab
// stalled, a non-finite value) is put on a list; the block elimination of k_newton.cuh then
// solves the listed regions from the start, with its own iteration cap and statistics.
#pragma once

#include <cuda_runtime.h>

#include "k_nl_lines.cuh"
#include "ridg_internal.h"

namespace ridg {
namespace mf {

using namespace nl;

// 1D tables, passed by value (constant bank): the FP64 residual rule, and
template <int NB>
struct Tab : nl::Rule<NB> {
  double Mt[NB][NB];   // time operator
  // the NB-point rule of the linearised operator
  float N[NB][NB];     // [b][n] phi_b(x_n)
  float M[NB][NB];     // [b][n] w_n / 2 phi_b(x_n): node values to modes
  float TN[NB][NB];    // [n][a] node values of (time operator)^-1 psi_a
  float Ti[NB][NB];    // [n][n'] inverse time operator on node values
  float D[NB][NB];     // [n][q] w_q sum_b phi_b(x_n) phi_b'(x_q)
  float E[2][NB];      // [side][n] sum_b phi_b(x_n) phi_b(+-1)
  float L[2][NB];      // [side][n] w_n / 2 E: trace of node values
};

template <int NB, int MV, bool F64 = false>
struct Cfg {
  static constexpr int THS = NB * NB, THT = NB * THS, BS = MV * THT, C = 9 * MV;
  static constexpr int NQ = residual_points(NB);
  static constexpr int COL = 9 * THS;               // columns (cell, y, x) of the region
  static constexpr int NT = (COL + 31) / 32 * 32, NW = NT / 32;
  static constexpr int VT = NB * MV;                // values per column
  static constexpr int FL = 24 * NB;                // face lines: 24 faces, NB lines each
  static constexpr int NG = MV == 1 ? 1 : 2;        // Burgers: one flux for both directions
  static_assert(FL <= NT, "one thread per face line");
  // CTAs per SM that the registers are held to, the best of a sweep for every degree and
  // precision (predictions with one CTA fewer / these / one more, in us.  FP32 solves: Burgers Q1
  // 128 x 120 573 / 554 / 572, Q2 96 x 100 1231 / 1136 / 1158, Q3 72 x 64 1277 / 1232 / 1236, Q4 60 x 50
  // 2868 / 2203 / 2249, Euler Q1 90 x 96 1245 / 1164 / 1217, Q2 96^2 5354 / 4559 / 5050; FP64: Burgers Q4
  // 7368 / 5690 / 6467, Euler Q2 15665 / 15676 / 18090, the others within 3% but for Q2's 2770 /
  // 2621 / 2646).  They cost 76 to 356 bytes of spills for Euler Q2, Burgers Q3 and Q4, and Euler Q1
  // in FP64.
  static constexpr int MINB = MV == 4 ? (NB == 2 ? 5 : F64 ? 2 : 3) : (NB == 2 ? 9 : NB == 3 ? 5 : NB == 4 ? 6 : 2);
  // FP64 arena: B1, B2 (line buffers), face fluxes; the face traces share B2
  static constexpr int nB = C * NB * NQ * NQ, nTr = 4 * C * NB * NQ, nH = 24 * MV * NB * NQ;
  static constexpr int nB2 = nB > nTr ? nB : nTr;
  // FP64 linear solves: the rule of the Jacobian (2M + 1 points of the quasi-quadrature-free
  // form; Burgers: exact with the residual's), the lines of two fields and the face fluxes
  static constexpr int NP = MV == 1 ? NQ : 2 * NB - 1;
  static constexpr int jB = C * NB * NP * NP, jTr = 4 * C * NB * NP, jH = 24 * MV * NB * NP;
  static constexpr int nLin = 2 * (jB > jTr ? jB : jTr) + jH;
  static constexpr int nRes = nB + nB2 + nH, nArena64 = F64 && nLin > nRes ? nLin : nRes;
  // FP32 arena: the vector, its fluxes, the face fluxes
  static constexpr int nP = VT * COL, nF = 24 * VT * NB;
  static constexpr int nArena32 = (1 + NG) * nP + nF;
  static constexpr size_t arena = nArena64 * 8 > nArena32 * 4 ? nArena64 * 8 : nArena32 * 4;
  static constexpr size_t oR = 8 * 9 * BS, oZ = 2 * oR, oD = oZ + (F64 ? oR : 0),
                          oQ = oD + (F64 ? oR : 0), oRed = oQ + 8 * C * THS, oArena = (oRed + 4 * 2 * 4 * NW + 15) / 16 * 16;
  static constexpr size_t bytes = oArena + arena;
};

// the cells left and right of region face f (dd * 12 + row * 4 + pos), -1 outside
__device__ __forceinline__ void face_cells(int f, int& dd, int& cl, int& cr) {
  dd = f >= 12;
  const int k = f - 12 * dd, row = k >> 2, pos = k & 3;
  cl = pos > 0 ? (dd ? (pos - 1) * 3 + row : row * 3 + pos - 1) : -1;
  cr = pos < 3 ? (dd ? pos * 3 + row : row * 3 + pos) : -1;
}

// body(line, time point, whether it counts) for LINES time lines of two points, a lane pair per
// line; whole warps take part (lanes past the end repeat the last line and must not write)
template <int LINES, int NT, class F>
__device__ __forceinline__ void time_pairs(F body) {
  for (int i0 = threadIdx.x & ~31; i0 < 2 * LINES; i0 += NT) {
    const int i = i0 + (threadIdx.x & 31), line = i >> 1;
    body(line < LINES ? line : LINES - 1, i & 1, line < LINES);
  }
}

// mode q of the two-point line whose values the lane pair holds (q: this lane's point)
__device__ __forceinline__ double pair_mode(const nl::Rule<2>& T, double f, int q) {
  const double o = __shfl_xor_sync(0xffffffffu, f, 1);
  const double so = __hiloint2double(__double2hiint(o) ^ (q << 31), __double2loint(o));  // -+o
  return (q ? -T.wV[1][0] : T.wV[0][0]) * (f + so);
}

// ---------------------------------------------------------------------------------------
// residual of eq. pred_full_system for the 9 region cells in FP64 (the sums of
// newton::residual).  FIRST: at the initial iterate (constant in time; the time term and the
// source cancel), where the face speeds alpha[24] are also taken and frozen.
// ---------------------------------------------------------------------------------------
template <int NB, int MV, int FLUX, bool FIRST>
__device__ void residual(const Tab<NB>& T, const double* Ws, const double* Qs, double* Rs,
                         double* alpha, double* arena, const double* lam, double g) {
  using K = Cfg<NB, MV>;
  constexpr int NQ = K::NQ, C = K::C, NT = K::NT, THS = K::THS, NA = FIRST ? 1 : NB,
                NX = NQ * NQ;
  const int tid = threadIdx.x;
  double* B1 = arena;              // [c][a][y][x], y and x with NQ slots
  double* B2 = B1 + K::nB;
  double* Tr = B2;                 // [dd][side][c][a][NQ]
  double* Hf = B2 + K::nB2;        // [face][j][a][NQ]
  // x lines: values at the x points, and the x traces (side 0: +1, 1: -1)
  for (int i = tid; i < C * NA * NB; i += NT) {
    const int c = i / (NA * NB), a = (i / NB) % NA, y = i % NB;
    const double* src = Ws + (c * NB + a) * THS + y * NB;
    double m[NB], v[NQ];
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = src[b];
    interp(T, m, v);
    double* dst = B1 + ((c * NB + a) * NQ + y) * NQ;
#pragma unroll
    for (int q = 0; q < NQ; ++q) dst[q] = v[q];
    double e, o;
    traces(T, m, 1, e, o);
    Tr[((0 * C + c) * NB + a) * NQ + y] = e + o;
    Tr[((1 * C + c) * NB + a) * NQ + y] = e - o;
  }
  // y traces
  for (int i = tid; i < C * NA * NB; i += NT) {
    const int c = i / (NA * NB), a = (i / NB) % NA, x = i % NB;
    const double* src = Ws + (c * NB + a) * THS + x;
    double e, o;
    traces(T, src, NB, e, o);
    Tr[((2 * C + c) * NB + a) * NQ + x] = e + o;
    Tr[((3 * C + c) * NB + a) * NQ + x] = e - o;
  }
  __syncthreads();
  // y lines, and the traces along their faces (in place: a line is read and written by the
  // same thread)
  for (int i = tid; i < C * NA * NQ; i += NT) {
    const int c = i / (NA * NQ), a = (i / NQ) % NA, x = i % NQ;
    double* p = B1 + (c * NB + a) * NX + x;
    double m[NB], v[NQ];
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = p[b * NQ];
    interp(T, m, v);
#pragma unroll
    for (int q = 0; q < NQ; ++q) p[q * NQ] = v[q];
  }
  for (int i = tid; i < 4 * C * NA; i += NT) {
    double* p = Tr + (i / NA * NB + i % NA) * NQ;
    double m[NB], v[NQ];
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = p[b];
    interp(T, m, v);
#pragma unroll
    for (int q = 0; q < NQ; ++q) p[q] = v[q];
  }
  __syncthreads();
  if constexpr (FIRST) {
    // Rusanov speeds: the largest of both sides over the face's points (time-constant)
    for (int f = tid; f < 24; f += NT) {
      int dd, cl, cr;
      face_cells(f, dd, cl, cr);
      double s = 0.0;
      if (cl >= 0 && cr >= 0) {
        for (int q = 0; q < NQ; ++q) {
          double wl[MV], wr[MV];
          for (int j = 0; j < MV; ++j) {
            wl[j] = Tr[((dd * 2 * C + cl * MV + j) * NB) * NQ + q];
            wr[j] = Tr[(((dd * 2 + 1) * C + cr * MV + j) * NB) * NQ + q];
          }
          s = fmax(s, fmax(nlflux::speed<FLUX>(wl, dd, g), nlflux::speed<FLUX>(wr, dd, g)));
        }
      }
      alpha[f] = s;
    }
    __syncthreads();
  }
  // Degree 1: the 36 volume and 48 face time lines fill little over half of two warps, whose
  // idle lanes cost the FP64 pipe as much as busy ones; a lane pair shares a line, one of its two
  // time points each, and exchanges the fluxes (Euler 67 x 90, four steps: 3.79 -> 3.65 ms).
  constexpr bool PAIR = NB == 2 && !FIRST;
  // time lines of the face points: both traces, the face flux, projected onto the time modes
  if constexpr (PAIR) {
    time_pairs<24 * NQ, NT>([&](int f_qo, int q, bool act) {
      const int f = f_qo / NQ, qo = f_qo - f * NQ;
      int dd, cl, cr;
      face_cells(f, dd, cl, cr);
      const double* tl = Tr + (dd * 2 * C + (cl < 0 ? cr : cl) * MV) * NB * NQ + qo;
      const double* tr = Tr + ((dd * 2 + 1) * C + (cr < 0 ? cl : cr) * MV) * NB * NQ + qo;
      const double al = 0.5 * alpha[f], v1 = q ? -T.V[1][0] : T.V[1][0];
      double wl[MV], wr[MV], fl[MV], fr[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        wl[j] = fma(v1, tl[(j * NB + 1) * NQ], tl[j * NB * NQ]);
        wr[j] = fma(v1, tr[(j * NB + 1) * NQ], tr[j * NB * NQ]);
      }
      if (cl >= 0) flux1<FLUX>(wl, dd, fl, g);
      if (cr >= 0) flux1<FLUX>(wr, dd, fr, g);
      double* h = Hf + (f * MV * NB + q) * NQ + qo;
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        const double fh = cl < 0 ? fr[j] : cr < 0 ? fl[j]
                          : fma(0.5, fl[j] + fr[j], -al * (wr[j] - wl[j]));
        const double m = pair_mode(T, fh, q);
        if (act) h[j * NB * NQ] = m;
      }
    });
  } else
  for (int i = tid; i < 24 * NQ; i += NT) {
    const int f = i / NQ, qo = i - f * NQ;
    int dd, cl, cr;
    face_cells(f, dd, cl, cr);
    const double* tl = Tr + (dd * 2 * C + (cl < 0 ? cr : cl) * MV) * NB * NQ + qo;
    const double* tr = Tr + ((dd * 2 + 1) * C + (cr < 0 ? cl : cr) * MV) * NB * NQ + qo;
    const double al = 0.5 * alpha[f];
    double* h = Hf + f * MV * NB * NQ + qo;
    double ml[MV][NA], mr[MV][NA], acc[MV][NA];
#pragma unroll
    for (int j = 0; j < MV; ++j)
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        ml[j][a] = tl[(j * NB + a) * NQ];
        mr[j][a] = tr[(j * NB + a) * NQ];
        acc[j][a] = 0.0;
      }
#pragma unroll
    for (int q = 0; q < (FIRST ? 1 : NQ); ++q) {
      double wl[MV], wr[MV], fl[MV], fr[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        wl[j] = ml[j][0];
        wr[j] = mr[j][0];
#pragma unroll
        for (int a = 1; a < NA; ++a) {
          wl[j] = fma(vq(T, a, q), ml[j][a], wl[j]);
          wr[j] = fma(vq(T, a, q), mr[j][a], wr[j]);
        }
      }
      if (cl >= 0) flux1<FLUX>(wl, dd, fl, g);
      if (cr >= 0) flux1<FLUX>(wr, dd, fr, g);
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        // region boundary: the interior trace alone
        const double fh = cl < 0 ? fr[j] : cr < 0 ? fl[j]
                          : fma(0.5, fl[j] + fr[j], -al * (wr[j] - wl[j]));
        if constexpr (FIRST) {
          acc[j][0] = 2.0 * fh;
        } else {
#pragma unroll
          for (int a = 0; a < NA; ++a) acc[j][a] = fma(wvq(T, a, q), fh, acc[j][a]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < MV; ++j)
#pragma unroll
      for (int a = 0; a < NA; ++a) h[(j * NB + a) * NQ] = acc[j][a];
  }
  __syncthreads();  // the traces (in B2) are consumed
  // time lines of the volume points: values, both fluxes, projected onto the time modes
  if constexpr (PAIR) {
    time_pairs<9 * NX, NT>([&](int i, int q, bool act) {
      const int r = i / NX, yx = i - r * NX;
      double* p1 = B1 + r * MV * NB * NX + yx;
      double* p2 = B2 + r * MV * NB * NX + yx;
      const double v1 = q ? -T.V[1][0] : T.V[1][0];
      double w[MV], fx[MV], fy[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) w[j] = fma(v1, p1[(j * NB + 1) * NX], p1[j * NB * NX]);
      flux2<FLUX>(w, fx, fy, g);
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        fx[j] = pair_mode(T, fx[j], q);
        if constexpr (K::NG == 2) fy[j] = pair_mode(T, fy[j], q);
      }
      __syncwarp();  // p1 is read by both lanes of a line
      if (act) {
#pragma unroll
        for (int j = 0; j < MV; ++j) {
          p1[(j * NB + q) * NX] = fx[j];
          if constexpr (K::NG == 2) p2[(j * NB + q) * NX] = fy[j];
        }
      }
    });
  } else
  for (int i = tid; i < 9 * NX; i += NT) {
    const int r = i / NX, yx = i - r * NX;
    double* p1 = B1 + r * MV * NB * NX + yx;
    double* p2 = B2 + r * MV * NB * NX + yx;
    if constexpr (FIRST) {
      double w[MV], fx[MV], fy[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) w[j] = p1[j * NB * NX];
      flux2<FLUX>(w, fx, fy, g);
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        p1[j * NB * NX] = 2.0 * fx[j];
        if constexpr (K::NG == 2) p2[j * NB * NX] = 2.0 * fy[j];
      }
    } else if constexpr (MV == 1) {
      double m[NB], v[NQ];
#pragma unroll
      for (int a = 0; a < NB; ++a) m[a] = p1[a * NX];
      interp(T, m, v);
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = 0.5 * v[q] * v[q];
      project<false>(T, v, m);
#pragma unroll
      for (int a = 0; a < NB; ++a) p1[a * NX] = m[a];
    } else {
      double m[MV][NB], ax[MV][NB], ay[MV][NB];
#pragma unroll
      for (int j = 0; j < MV; ++j)
#pragma unroll
        for (int a = 0; a < NB; ++a) {
          m[j][a] = p1[(j * NB + a) * NX];
          ax[j][a] = ay[j][a] = 0.0;
        }
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        double w[MV], fx[MV], fy[MV];
#pragma unroll
        for (int j = 0; j < MV; ++j) {
          w[j] = m[j][0];
#pragma unroll
          for (int a = 1; a < NB; ++a) w[j] = fma(vq(T, a, q), m[j][a], w[j]);
        }
        flux2<FLUX>(w, fx, fy, g);
#pragma unroll
        for (int j = 0; j < MV; ++j)
#pragma unroll
          for (int a = 0; a < NB; ++a) {
            ax[j][a] = fma(wvq(T, a, q), fx[j], ax[j][a]);
            ay[j][a] = fma(wvq(T, a, q), fy[j], ay[j][a]);
          }
      }
#pragma unroll
      for (int j = 0; j < MV; ++j)
#pragma unroll
        for (int a = 0; a < NB; ++a) {
          p1[(j * NB + a) * NX] = ax[j][a];
          p2[(j * NB + a) * NX] = ay[j][a];
        }
    }
  }
  __syncthreads();
  // y lines back: the x flux with phi_y, the y flux with phi_y'; the face lines along them
  for (int i = tid; i < C * NA * NQ; i += NT) {
    const int c = i / (NA * NQ), a = (i / NQ) % NA, x = i % NQ;
    double* p1 = B1 + (c * NB + a) * NX + x;
    double* p2 = B2 + (c * NB + a) * NX + x;
    double f[NQ], o1[NB], o2[NB];
#pragma unroll
    for (int q = 0; q < NQ; ++q) f[q] = p1[q * NQ];
    project<false>(T, f, o1);
    if constexpr (K::NG == 2) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) f[q] = p2[q * NQ];
    }
    project<true>(T, f, o2);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      p1[b * NQ] = o1[b];
      p2[b * NQ] = o2[b];
    }
  }
  for (int i = tid; i < 24 * MV * NA; i += NT) {
    double* p = Hf + (i / NA * NB + i % NA) * NQ;
    double f[NQ], o[NB];
#pragma unroll
    for (int q = 0; q < NQ; ++q) f[q] = p[q];
    project<false>(T, f, o);
#pragma unroll
    for (int b = 0; b < NB; ++b) p[b] = o[b];
  }
  __syncthreads();
  // x lines back, and R = time term - source - volume + faces
  const double l0 = 0.25 * lam[0], l1 = 0.25 * lam[1];
  for (int i = tid; i < C * NB * NB; i += NT) {
    const int c = i / (NB * NB), a = (i / NB) % NB, y = i % NB;
    double* out = Rs + (c * NB + a) * THS + y * NB;
    if (FIRST && a > 0) {
#pragma unroll
      for (int b = 0; b < NB; ++b) out[b] = 0.0;
      continue;
    }
    const int r = c / MV, j = c - r * MV, ry = r / 3, rx = r - 3 * ry;
    const double* p1 = B1 + ((c * NB + a) * NQ + y) * NQ;
    const double* p2 = B2 + ((c * NB + a) * NQ + y) * NQ;
    double f[NQ], ox[NB], oy[NB];
#pragma unroll
    for (int q = 0; q < NQ; ++q) f[q] = p1[q];
    project<true>(T, f, ox);
#pragma unroll
    for (int q = 0; q < NQ; ++q) f[q] = p2[q];
    project<false>(T, f, oy);
    const double* hx = Hf + (((ry * 4 + rx) * MV + j) * NB + a) * NQ;         // left face
    const double* hy = Hf + (((12 + rx * 4 + ry) * MV + j) * NB + a) * NQ;    // lower face
    const double hl = hx[y], hr = hx[MV * NB * NQ + y];
    const double sx = hr - hl, dx = hr + hl;  // even / odd x modes: ep (hr -+ hl)
    const double ey = T.ep[y];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const double hb = hy[b], ht = hy[MV * NB * NQ + b];
      const double fy = (y & 1) ? ht + hb : ht - hb;
      double acc = l0 * fma(T.ep[b], (b & 1) ? dx : sx, -ox[b]);
      acc = fma(l1, fma(ey, fy, -oy[b]), acc);
      if constexpr (!FIRST) {
        const double* w = Ws + c * K::THT + y * NB + b;
#pragma unroll
        for (int e = 0; e < NB; ++e) acc = fma(T.Mt[a][e], w[e * THS], acc);
        // psi_a(-1) Q
        acc = fma((a & 1) ? T.ep[a] : -T.ep[a], Qs[c * THS + y * NB + b], acc);
      }
      out[b] = acc;
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------------------
// Rs -= J z in FP64: the linearised residual at W (the sums of `residual` with F'(w) z for the
// fluxes), by the rule T of the Jacobian.  Euler: 2M + 1 points per dimension, on which the
// quasi-quadrature-free Jacobian's projection onto degree 2M is interpolation and its triple
// products are exact -- the same matrix as the block elimination's.
// ---------------------------------------------------------------------------------------
template <int NB, int MV, int FLUX, int NP>
__device__ void linear_update(const Rule<NB, NP>& T, const double (&Mt)[NB][NB], const double* Ws,
                              const double* Zs, double* Rs, const double* alpha, double* arena,
                              const double* lam, double g) {
  using K = Cfg<NB, MV, true>;
  constexpr int C = K::C, NT = K::NT, THS = K::THS, NX = NP * NP;
  const int tid = threadIdx.x;
  double* B0 = arena;                                      // lines of w, then the x flux
  double* B1 = B0 + (K::jB > K::jTr ? K::jB : K::jTr);     // lines of z, then the y flux
  double* Hf = B1 + (K::jB > K::jTr ? K::jB : K::jTr);     // [face][j][a][NP]
  // face traces of both fields, [dd][side][c][a][NP] in B0 (w) and B1 (z)
  for (int i = tid; i < 4 * C * NB * NB; i += NT) {
    const int fd = i / (C * NB * NB), k = i - fd * (C * NB * NB), ca = k / NB, o = k - ca * NB;
    const int dd = fd & 1;
    const double* src = (fd & 2 ? Zs : Ws) + ca * THS + (dd ? o : o * NB);
    double* tr = (fd & 2 ? B1 : B0) + (dd * 2 * C * NB + ca) * NP + o;
    double e, od;
    traces(T, src, dd ? NB : 1, e, od);
    tr[0] = e + od;
    tr[C * NB * NP] = e - od;
  }
  __syncthreads();
  for (int i = tid; i < 8 * C * NB; i += NT) {
    double* p = (i < 4 * C * NB ? B0 + i * NP : B1 + (i - 4 * C * NB) * NP);
    double m[NB], v[NP];
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = p[b];
    interp(T, m, v);
#pragma unroll
    for (int q = 0; q < NP; ++q) p[q] = v[q];
  }
  __syncthreads();
  for (int i = tid; i < 24 * NP; i += NT) {
    const int f = i / NP, qo = i - f * NP;
    int dd, cl, cr;
    face_cells(f, dd, cl, cr);
    const int tl = (dd * 2 * C + (cl < 0 ? cr : cl) * MV) * NB * NP + qo;
    const int tr = ((dd * 2 + 1) * C + (cr < 0 ? cl : cr) * MV) * NB * NP + qo;
    const double al = 0.5 * alpha[f];
    double acc[MV][NB];
#pragma unroll
    for (int j = 0; j < MV; ++j)
#pragma unroll
      for (int a = 0; a < NB; ++a) acc[j][a] = 0.0;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      double wl[MV], wr[MV], zl[MV], zr[MV], fl[MV], fr[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        wl[j] = B0[tl + j * NB * NP];
        wr[j] = B0[tr + j * NB * NP];
        zl[j] = B1[tl + j * NB * NP];
        zr[j] = B1[tr + j * NB * NP];
#pragma unroll
        for (int a = 1; a < NB; ++a) {
          const double v = vq(T, a, q);
          const int at = (j * NB + a) * NP;
          wl[j] = fma(v, B0[tl + at], wl[j]);
          wr[j] = fma(v, B0[tr + at], wr[j]);
          zl[j] = fma(v, B1[tl + at], zl[j]);
          zr[j] = fma(v, B1[tr + at], zr[j]);
        }
      }
      if (cl >= 0) dflux1<FLUX>(wl, zl, dd, fl, g);
      if (cr >= 0) dflux1<FLUX>(wr, zr, dd, fr, g);
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        const double fh = cl < 0 ? fr[j] : cr < 0 ? fl[j]
                          : fma(0.5, fl[j] + fr[j], -al * (zr[j] - zl[j]));
#pragma unroll
        for (int a = 0; a < NB; ++a) acc[j][a] = fma(wvq(T, a, q), fh, acc[j][a]);
      }
    }
    double* h = Hf + f * MV * NB * NP + qo;
#pragma unroll
    for (int j = 0; j < MV; ++j)
#pragma unroll
      for (int a = 0; a < NB; ++a) h[(j * NB + a) * NP] = acc[j][a];
  }
  __syncthreads();
  // volume: x lines, y lines of both fields
  for (int i = tid; i < 2 * C * NB * NB; i += NT) {
    const bool z = i >= C * NB * NB;
    const int k = z ? i - C * NB * NB : i, ca = k / NB, y = k - ca * NB;
    const double* src = (z ? Zs : Ws) + ca * THS + y * NB;
    double* dst = (z ? B1 : B0) + (ca * NP + y) * NP;
    double m[NB], v[NP];
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = src[b];
    interp(T, m, v);
#pragma unroll
    for (int q = 0; q < NP; ++q) dst[q] = v[q];
  }
  __syncthreads();
  for (int i = tid; i < 2 * C * NB * NP; i += NT) {
    const bool z = i >= C * NB * NP;
    const int k = z ? i - C * NB * NP : i, ca = k / NP;
    double* p = (z ? B1 : B0) + ca * NX + (k - ca * NP);
    double m[NB], v[NP];
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = p[b * NP];
    interp(T, m, v);
#pragma unroll
    for (int q = 0; q < NP; ++q) p[q * NP] = v[q];
  }
  __syncthreads();
  for (int i = tid; i < 9 * NX; i += NT) {
    const int r = i / NX, at = r * MV * NB * NX + (i - r * NX);
    double* p0 = B0 + at;
    double* p1 = B1 + at;
    double ax[MV][NB], ay[MV][NB];
#pragma unroll
    for (int j = 0; j < MV; ++j)
#pragma unroll
      for (int a = 0; a < NB; ++a) ax[j][a] = ay[j][a] = 0.0;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      double w[MV], z[MV], fx[MV], fy[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        w[j] = p0[j * NB * NX];
        z[j] = p1[j * NB * NX];
#pragma unroll
        for (int a = 1; a < NB; ++a) {
          const double v = vq(T, a, q);
          w[j] = fma(v, p0[(j * NB + a) * NX], w[j]);
          z[j] = fma(v, p1[(j * NB + a) * NX], z[j]);
        }
      }
      dflux2<FLUX>(w, z, fx, fy, g);
#pragma unroll
      for (int j = 0; j < MV; ++j)
#pragma unroll
        for (int a = 0; a < NB; ++a) {
          ax[j][a] = fma(wvq(T, a, q), fx[j], ax[j][a]);
          if constexpr (MV > 1) ay[j][a] = fma(wvq(T, a, q), fy[j], ay[j][a]);
        }
    }
#pragma unroll
    for (int j = 0; j < MV; ++j)
#pragma unroll
      for (int a = 0; a < NB; ++a) {
        p0[(j * NB + a) * NX] = ax[j][a];
        if constexpr (MV > 1) p1[(j * NB + a) * NX] = ay[j][a];
      }
  }
  __syncthreads();
  for (int i = tid; i < C * NB * NP; i += NT) {
    const int ca = i / NP;
    double* p0 = B0 + ca * NX + (i - ca * NP);
    double* p1 = B1 + ca * NX + (i - ca * NP);
    double f[NP], o1[NB], o2[NB];
#pragma unroll
    for (int q = 0; q < NP; ++q) f[q] = p0[q * NP];
    project<false>(T, f, o1);
    if constexpr (MV > 1) {
#pragma unroll
      for (int q = 0; q < NP; ++q) f[q] = p1[q * NP];
    }
    project<true>(T, f, o2);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      p0[b * NP] = o1[b];
      p1[b * NP] = o2[b];
    }
  }
  for (int i = tid; i < 24 * MV * NB; i += NT) {
    double* p = Hf + i * NP;
    double f[NP], o[NB];
#pragma unroll
    for (int q = 0; q < NP; ++q) f[q] = p[q];
    project<false>(T, f, o);
#pragma unroll
    for (int b = 0; b < NB; ++b) p[b] = o[b];
  }
  __syncthreads();
  const double l0 = 0.25 * lam[0], l1 = 0.25 * lam[1];
  for (int i = tid; i < C * NB * NB; i += NT) {
    const int c = i / (NB * NB), a = (i / NB) % NB, y = i % NB;
    const int r = c / MV, j = c - r * MV, ry = r / 3, rx = r - 3 * ry;
    double* out = Rs + (c * NB + a) * THS + y * NB;
    const double* p0 = B0 + ((c * NB + a) * NP + y) * NP;
    const double* p1 = B1 + ((c * NB + a) * NP + y) * NP;
    double f[NP], ox[NB], oy[NB];
#pragma unroll
    for (int q = 0; q < NP; ++q) f[q] = p0[q];
    project<true>(T, f, ox);
#pragma unroll
    for (int q = 0; q < NP; ++q) f[q] = p1[q];
    project<false>(T, f, oy);
    const double* hx = Hf + (((ry * 4 + rx) * MV + j) * NB + a) * NP;
    const double* hy = Hf + (((12 + rx * 4 + ry) * MV + j) * NB + a) * NP;
    const double hl = hx[y], hr = hx[MV * NB * NP + y], ey = T.ep[y];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const double hb = hy[b], ht = hy[MV * NB * NP + b];
      const double fx = (b & 1) ? hr + hl : hr - hl, fy = (y & 1) ? ht + hb : ht - hb;
      double acc = l0 * fma(T.ep[b], fx, -ox[b]);
      acc = fma(l1, fma(ey, fy, -oy[b]), acc);
      const double* z = Zs + c * K::THT + y * NB + b;
#pragma unroll
      for (int e = 0; e < NB; ++e) acc = fma(Mt[a][e], z[e * THS], acc);
      out[b] -= acc;
    }
  }
  __syncthreads();
}

// (F' v) for primitives (u, v, H) and both directions, or one
struct Prim {
  float u, v, H;
};
__device__ __forceinline__ void euler_jv(const Prim& s, const float* d, float g1, float* gx,
                                         float* gy) {
  const float k = 0.5f * fmaf(s.u, s.u, s.v * s.v);
  const float dp = g1 * (fmaf(k, d[0], d[3]) - fmaf(s.u, d[1], s.v * d[2]));
  const float a = fmaf(-s.u, d[0], d[1]), b = fmaf(-s.v, d[0], d[2]), h = d[3] + dp;
  gx[0] = d[1];
  gx[1] = fmaf(s.u, d[1] + a, dp);
  gx[2] = fmaf(s.v, a, s.u * d[2]);
  gx[3] = fmaf(s.H, a, s.u * h);
  gy[0] = d[2];
  gy[1] = fmaf(s.u, b, s.v * d[1]);
  gy[2] = fmaf(s.v, d[2] + b, dp);
  gy[3] = fmaf(s.H, b, s.v * h);
}
__device__ __forceinline__ void euler_jv1(const Prim& s, const float* d, float g1, int dd,
                                          float* f) {
  const float k = 0.5f * fmaf(s.u, s.u, s.v * s.v);
  const float dp = g1 * (fmaf(k, d[0], d[3]) - fmaf(s.u, d[1], s.v * d[2]));
  const float un = dd ? s.v : s.u, dn = dd ? d[2] : d[1];
  const float a = fmaf(-un, d[0], dn);  // rho d(u_n)
  f[0] = dn;
  f[1] = fmaf(s.u, a, un * d[1]);
  f[2] = fmaf(s.v, a, un * d[2]);
  if (dd) f[2] += dp; else f[1] += dp;
  f[3] = fmaf(s.H, a, un * (d[3] + dp));
}
__device__ __forceinline__ Prim prim_of(const float* w, float g1) {
  Prim s;
  const float ir = 1.0f / w[0];
  s.u = w[1] * ir;
  s.v = w[2] * ir;
  const float p = g1 * (w[3] - 0.5f * fmaf(w[1], s.u, w[2] * s.v));
  s.H = (w[3] + p) * ir;
  return s;
}

// in-place transform of the x or y lines of P: out[i] = sum_b A(b, i) in[b], A = M[i][b] (to
// modes) or N[b][i] (to nodes)
template <int NB, int MV, bool TO_NODES>
__device__ __forceinline__ void lines(const Tab<NB>& T, float* P, bool ydir) {
  using K = Cfg<NB, MV>;
  for (int i = threadIdx.x; i < K::VT * 9 * NB; i += K::NT) {
    const int tj = i / (9 * NB), ro = i - tj * 9 * NB, r = ro / NB, o = ro - r * NB;
    const int st = ydir ? NB : 1;
    float* p = P + tj * K::COL + r * K::THS + (ydir ? o : o * NB);
    float in[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) in[b] = p[b * st];
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      float s = 0.f;
#pragma unroll
      for (int b = 0; b < NB; ++b) s = fmaf(TO_NODES ? T.N[b][n] : T.M[n][b], in[b], s);
      p[n * st] = s;
    }
  }
}

// modal FP64 field src 2^-ex to FP32 values at the x nodes, y and time still modal; TINY: scaled in
// FP64, where FP32 would lose the small values
template <int NB, int MV, bool TINY>
__device__ __forceinline__ void x_nodes(const Tab<NB>& T, const double* src, int ex, float* P) {
  using K = Cfg<NB, MV>;
  const float sf = TINY ? 1.f : scalbnf(1.f, -ex);
  const double sd = TINY ? pow2(-ex) : 1.0;
  for (int i = threadIdx.x; i < K::VT * 9 * NB; i += K::NT) {
    const int tj = i / (9 * NB), ro = i - tj * 9 * NB, r = ro / NB, y = ro - r * NB;
    const int a = tj / MV, j = tj - a * MV;
    const double* s = src + ((r * MV + j) * NB + a) * K::THS + y * NB;
    float in[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) in[b] = TINY ? (float)(s[b] * sd) : (float)s[b] * sf;
    float* p = P + tj * K::COL + r * K::THS + y * NB;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      float v = 0.f;
#pragma unroll
      for (int b = 0; b < NB; ++b) v = fmaf(T.N[b][n], in[b], v);
      p[n] = v;
    }
  }
}

// the same at the (y, x) nodes
template <int NB, int MV>
__device__ __forceinline__ void to_nodes(const Tab<NB>& T, const double* src, int ex, float* P) {
  if (ex >= -100) x_nodes<NB, MV, false>(T, src, ex, P); else x_nodes<NB, MV, true>(T, src, ex, P);
  __syncthreads();
  lines<NB, MV, true>(T, P, true);
  __syncthreads();
}

// The linearisation point of a thread: F' at the nodes of its column and at both sides of
// its face line (Burgers: the value; Euler: primitives).
template <int NB, int MV>
struct Lin {
  float w[NB], wl[NB], wr[NB];
};
template <int NB>
struct Lin<NB, 4> {
  Prim w[NB], wl[NB], wr[NB];
};

// Thread constants of the linearised operator: the thread's column (cell, y, x) and its
// face line.
template <int NB>
struct Rows {
  float dx[NB], dy[NB], xp, xm, yp, ym;  // -lam D rows, +-lam E of the column's node
  int gx, gy;                            // its x line (first node) and y line in a flux array
  int fx, fy;                            // its left / lower face value: (face * VT) * NB + line
  int dd, bl, br;                        // face line: direction, first nodes (-1: outside)
  float al;                              // alpha / 2
};

// out = (time operator)^-1 J v on node values, all 9 cells
template <int NB, int MV, int FLUX>
__device__ __forceinline__ void apply(const Tab<NB>& T, const Rows<NB>& R, const Lin<NB, MV>& S,
                                      const float (&v)[NB * MV], float (&out)[NB * MV], float* P,
                                      float* G, float* Fh, float g1) {
  using K = Cfg<NB, MV>;
  constexpr int VT = K::VT, COL = K::COL;
  const int tid = threadIdx.x;
  if (tid < COL) {
#pragma unroll
    for (int t = 0; t < NB; ++t) {
      if constexpr (MV == 1) {
        P[t * COL + tid] = v[t];
        G[t * COL + tid] = S.w[t] * v[t];
      } else {
        float gx[MV], gy[MV];
        euler_jv(S.w[t], v + t * MV, g1, gx, gy);
#pragma unroll
        for (int j = 0; j < MV; ++j) {
          P[(t * MV + j) * COL + tid] = v[t * MV + j];
          G[(t * MV + j) * COL + tid] = gx[j];
          G[K::nP + (t * MV + j) * COL + tid] = gy[j];
        }
      }
    }
  }
  __syncthreads();
  if (tid < K::FL) {
    const int st = R.dd ? NB : 1, f = tid / NB, o = tid - f * NB;
    float* h = Fh + f * VT * NB + o;
#pragma unroll
    for (int t = 0; t < NB; ++t) {
      float vl[MV], vr[MV], fl[MV], fr[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        vl[j] = vr[j] = 0.f;
        const float* p = P + (t * MV + j) * COL;
        if (R.bl >= 0)
#pragma unroll
          for (int n = 0; n < NB; ++n) vl[j] = fmaf(T.L[0][n], p[R.bl + n * st], vl[j]);
        if (R.br >= 0)
#pragma unroll
          for (int n = 0; n < NB; ++n) vr[j] = fmaf(T.L[1][n], p[R.br + n * st], vr[j]);
      }
      if constexpr (MV == 1) {
        fl[0] = S.wl[t] * vl[0];
        fr[0] = S.wr[t] * vr[0];
      } else {
        euler_jv1(S.wl[t], vl, g1, R.dd, fl);
        euler_jv1(S.wr[t], vr, g1, R.dd, fr);
      }
#pragma unroll
      for (int j = 0; j < MV; ++j)
        h[(t * MV + j) * NB] = R.bl < 0   ? fr[j]
                               : R.br < 0 ? fl[j]
                                          : fmaf(0.5f, fl[j] + fr[j], -R.al * (vr[j] - vl[j]));
    }
  }
  __syncthreads();
  if (tid < COL) {
    float acc[VT];
#pragma unroll
    for (int tj = 0; tj < VT; ++tj) {
      const float* gx = G + tj * COL + R.gx;
      const float* gy = G + (K::NG == 2 ? K::nP : 0) + tj * COL + R.gy;
      float s = 0.f;
#pragma unroll
      for (int n = 0; n < NB; ++n) s = fmaf(R.dx[n], gx[n], s);
#pragma unroll
      for (int n = 0; n < NB; ++n) s = fmaf(R.dy[n], gy[n * NB], s);
      const float* hx = Fh + R.fx + tj * NB;
      const float* hy = Fh + R.fy + tj * NB;
      s = fmaf(R.xm, hx[0], s);
      s = fmaf(R.xp, hx[VT * NB], s);
      s = fmaf(R.ym, hy[0], s);
      s = fmaf(R.yp, hy[VT * NB], s);
      acc[tj] = s;
    }
#pragma unroll
    for (int t = 0; t < NB; ++t)
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        float s = v[t * MV + j];
#pragma unroll
        for (int e = 0; e < NB; ++e) s = fmaf(T.Ti[t][e], acc[e * MV + j], s);
        out[t * MV + j] = s;
      }
  }
}

// Linear solves of a region (mixed) before it is left to the list; no more than the block
// elimination makes at the caller's cap (1 + kSweepsFp32 per factorisation, which is fewer at a
// cap of one), so that a region stopped by the cap there is not reported as converged here.
constexpr int kMaxSolves = 7;
constexpr int kMaxRefine = 8;   // FP32 solves per Newton iteration (FP64) before that
constexpr int kMaxInner = 32;   // BiCGStab iterations per solve

// The linearisation point at W: F' at the thread's nodes and at both sides of its face line.
template <int NB, int MV>
__device__ __forceinline__ void linearise(const Tab<NB>& T, const double* Ws, const Rows<NB>& R,
                                          Lin<NB, MV>& S, float* P, float g1) {
  using K = Cfg<NB, MV>;
  constexpr int VT = K::VT, COL = K::COL;
  const int tid = threadIdx.x;
  to_nodes<NB, MV>(T, Ws, 0, P);
  if (tid < COL) {
    float m[VT], w[VT];
#pragma unroll
    for (int tj = 0; tj < VT; ++tj) m[tj] = P[tj * COL + tid];
#pragma unroll
    for (int t = 0; t < NB; ++t)
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        float s = 0.f;
#pragma unroll
        for (int b = 0; b < NB; ++b) s = fmaf(T.N[b][t], m[b * MV + j], s);
        w[t * MV + j] = s;
      }
#pragma unroll
    for (int tj = 0; tj < VT; ++tj) P[tj * COL + tid] = w[tj];
#pragma unroll
    for (int t = 0; t < NB; ++t) {
      if constexpr (MV == 1) S.w[t] = w[t];
      else S.w[t] = prim_of(w + t * MV, g1);
    }
  }
  __syncthreads();
  if (tid < K::FL) {
    const int st = R.dd ? NB : 1;
    // outside the region the inner trace stands in (its flux is not used)
    const int bl = R.bl < 0 ? R.br : R.bl, br = R.br < 0 ? R.bl : R.br;
#pragma unroll
    for (int t = 0; t < NB; ++t) {
      float l[MV], r[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        const float* p = P + (t * MV + j) * COL;
        l[j] = r[j] = 0.f;
#pragma unroll
        for (int n = 0; n < NB; ++n) {
          l[j] = fmaf(T.L[R.bl < 0][n], p[bl + n * st], l[j]);
          r[j] = fmaf(T.L[R.br < 0 ? 0 : 1][n], p[br + n * st], r[j]);
        }
      }
      if constexpr (MV == 1) {
        S.wl[t] = l[0];
        S.wr[t] = r[0];
      } else {
        S.wl[t] = prim_of(l, g1);
        S.wr[t] = prim_of(r, g1);
      }
    }
  }
  __syncthreads();
}

// J z = 2^-ex Rs by BiCGStab in FP32 to a relative residual of about atol / |2^-ex Rs| within
// [rmin, rmax]; the modes of z are left in P (all threads may read them) and the relative
// residual reached in `ratio`.  False if it stalled.
template <int NB, int MV, int FLUX>
__device__ __forceinline__ bool bicgstab(const Tab<NB>& T, const Rows<NB>& R,
                                         const Lin<NB, MV>& S, const double* Rs, int ex,
                                         float atol, float rmin, float rmax, float* P, float* G,
                                         float* Fh, float* red, int& buf, float g1,
                                         float& ratio) {
  using K = Cfg<NB, MV>;
  constexpr int VT = K::VT, COL = K::COL, NW = K::NW;
  const int tid = threadIdx.x;
  // right-hand side: node values of (time operator)^-1 R, scaled
  to_nodes<NB, MV>(T, Rs, ex, P);
  float r[VT], rh[VT], p[VT], v[VT], t[VT], x[VT];
  float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < VT; ++k) r[k] = p[k] = v[k] = t[k] = x[k] = 0.f;
  if (tid < COL) {
    float m[VT];
#pragma unroll
    for (int tj = 0; tj < VT; ++tj) m[tj] = P[tj * COL + tid];
#pragma unroll
    for (int n = 0; n < NB; ++n)
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        float s = 0.f;
#pragma unroll
        for (int b = 0; b < NB; ++b) s = fmaf(T.TN[n][b], m[b * MV + j], s);
        r[n * MV + j] = s;
      }
  }
#pragma unroll
  for (int k = 0; k < VT; ++k) {
    rh[k] = p[k] = r[k];
    s4[0] = fmaf(r[k], r[k], s4[0]);
  }
  {
    float s1[1] = {s4[0]};
    reduce<NW, 1, false>(s1, red, buf);
    s4[0] = s1[0];
  }
  const float bb = s4[0];
  const float bmean = sqrtf(bb / (9 * K::BS));
  const float tol = fminf(rmax, fmaxf(rmin, atol / bmean));
  const float stop = tol * tol * bb;
  float rho = bb, rr = bb, hh = bb;  // <rh, r>, |r|^2, |rh|^2
#pragma unroll 1
  for (int k = 0; k < 2 * kMaxInner && rr > stop; ++k) {
    float s1[1] = {0.f};
    if (k == kMaxInner) {
      if (rr <= 0.1f * bb) break;
      // stalled (a few regions in ten thousand, with right-hand sides of round-off size): again
      // from r with another shadow vector, every second column of r
#pragma unroll
      for (int q = 0; q < VT; ++q) {
        p[q] = r[q];
        rh[q] = (tid & 1) ? 0.f : r[q];
        s1[0] = fmaf(rh[q], r[q], s1[0]);
      }
      reduce<NW, 1, false>(s1, red, buf);
      rho = hh = s1[0];
      s1[0] = 0.f;
    }
    apply<NB, MV, FLUX>(T, R, S, p, v, P, G, Fh, g1);
    if (tid < COL)
#pragma unroll
      for (int q = 0; q < VT; ++q) s1[0] = fmaf(rh[q], v[q], s1[0]);
    reduce<NW, 1, false>(s1, red, buf);
    const float al = rho / s1[0];
#pragma unroll
    for (int q = 0; q < VT; ++q) r[q] = fmaf(-al, v[q], r[q]);  // s of the method
    apply<NB, MV, FLUX>(T, R, S, r, t, P, G, Fh, g1);
    s4[0] = s4[1] = s4[2] = s4[3] = 0.f;
    if (tid < COL)
#pragma unroll
      for (int q = 0; q < VT; ++q) {
        s4[0] = fmaf(t[q], r[q], s4[0]);
        s4[1] = fmaf(t[q], t[q], s4[1]);
        s4[2] = fmaf(rh[q], t[q], s4[2]);
        s4[3] = fmaf(r[q], r[q], s4[3]);
      }
    reduce<NW, 4, false>(s4, red, buf);
    const float om = s4[1] > 0.f ? s4[0] / s4[1] : 0.f;
#pragma unroll
    for (int q = 0; q < VT; ++q) {
      x[q] = fmaf(al, p[q], fmaf(om, r[q], x[q]));
      r[q] = fmaf(-om, t[q], r[q]);
    }
    rr = fmaxf(0.f, s4[3] - om * s4[0]);
    if (!(fabsf(al) < 1e30f) || !(rr < 1e30f)) return false;
    const float rho1 = -om * s4[2];  // <rh, r>, as <rh, s> = 0
    if (rho1 * rho1 <= 1e-5f * rr * hh) {
      // r is all but orthogonal to the shadow vector, and the method about to stall: start anew
      // from r
#pragma unroll
      for (int q = 0; q < VT; ++q) rh[q] = p[q] = r[q];
      rho = hh = rr;
      continue;
    }
    const float be = rho1 / rho * (al / om);
    rho = rho1;
#pragma unroll
    for (int q = 0; q < VT; ++q) p[q] = fmaf(be, fmaf(-om, v[q], p[q]), r[q]);
  }
  // (what a slow solve leaves is the next one's right-hand side)
  if (rr > 0.1f * bb) return false;
  ratio = bb > 0.f ? sqrtf(rr / bb) : 0.f;
  // the modes of x
  __syncthreads();
  if (tid < COL) {
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        float s = 0.f;
#pragma unroll
        for (int n = 0; n < NB; ++n) s = fmaf(T.M[b][n], x[n * MV + j], s);
        P[(b * MV + j) * COL + tid] = s;
      }
  }
  __syncthreads();
  lines<NB, MV, false>(T, P, true);
  __syncthreads();
  lines<NB, MV, false>(T, P, false);
  __syncthreads();
  return true;
}

// a block's largest |x| by its high word, rounded down; 3e38 if not finite or above 1e30
__device__ __forceinline__ float max_of_hi(int hi) {
  return hi < kHi1e30 ? __double2float_rd(__hiloint2double(hi, 0)) : 3e38f;
}
template <int NW>
__device__ __forceinline__ float block_max(MaxAbs m, float* red, int& buf) {
  return max_of_hi(block_max_hi<NW>(m, red, buf));
}

// the largest |Rs| and its exponent ex; false if unusable
template <int NB, int MV>
__device__ __forceinline__ bool rhs_scale(const double* Rs, float* red, int& buf, float& rmax,
                                          int& ex) {
  using K = Cfg<NB, MV>;
  MaxAbs m;
  for (int i = threadIdx.x; i < 9 * K::BS; i += K::NT) m.add(Rs[i]);
  const int hi = block_max_hi<K::NW>(m, red, buf);
  rmax = max_of_hi(hi);
  ex = exponent_of(hi);
  return hi < kHi1e30;
}

// index in P of the modal entry i of a region field ([cell][variable][time][y, x])
template <int NB, int MV>
__device__ __forceinline__ int p_index(int i) {
  using K = Cfg<NB, MV>;
  const int c = i / K::THT, m = i - c * K::THT, a = m / K::THS, s = m - a * K::THS;
  const int r = c / MV, j = c - r * MV;
  return (a * MV + j) * K::COL + r * K::THS + s;
}

// F64 = false (the mixed precisions): chord iteration -- one FP32 solve per FP64 residual, the
// linearisation renewed where it no longer contracts well.  F64 = true: Newton with every
// linear system solved to FP64 accuracy, by FP32 solves refined against its FP64 residual, so
// that the iterates are the block elimination's to round-off.
template <int NB, int MV, int FLUX, bool F64, bool BATCH>
__global__ void __launch_bounds__((Cfg<NB, MV, F64>::NT), (Cfg<NB, MV, F64>::MINB))
    newton_mf_kernel(const NewtonMfArgs a, const Tab<NB> T,
                     const Rule<NB, Cfg<NB, MV, F64>::NP> TJ) {
  using K = Cfg<NB, MV, F64>;
  constexpr int VT = K::VT, COL = K::COL, NT = K::NT, NW = K::NW, THS = K::THS, BS = K::BS;
  extern __shared__ __align__(16) unsigned char smem[];
  double* Ws = (double*)smem;
  double* Rs = (double*)(smem + K::oR);
  double* Zs = (double*)(smem + K::oZ);  // F64: the last FP32 solve's result
  double* Ds = (double*)(smem + K::oD);  // F64: the Newton update
  double* Qs = (double*)(smem + K::oQ);
  __shared__ double alpha[24];
  float* red = (float*)(smem + K::oRed);
  double* arena = (double*)(smem + K::oArena);
  float* P = (float*)arena;
  float* G = P + K::nP;
  float* Fh = G + K::NG * K::nP;
  const int tid = threadIdx.x;
  const long long eg = blockIdx.x;
  // the region's instance (batched launch: the last whose first region is <= eg)
  const double* Qg = a.Q;
  double* Wg = a.W;
  int* stats = a.stats;
  unsigned long long* itot = a.iters_total;
  int nx = a.nx, ny = a.ny;
  long long e = eg;
  double lam[2] = {a.lam[0], a.lam[1]};
  if constexpr (BATCH) {
    int lo = 0, hi = a.ninst - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.inst[mid].cell0 <= eg) lo = mid; else hi = mid - 1;
    }
    const NlInst& in = a.inst[lo];
    Qg = in.Q;
    Wg = in.W;
    stats = in.stats;
    itot = in.iters_total;
    nx = in.nx;
    ny = in.ny;
    e = eg - in.cell0;
    lam[0] = in.lam[0];
    lam[1] = in.lam[1];
  }
  const unsigned ue = (unsigned)e, uy = ue / (unsigned)nx;
  const int ix = (int)(ue - uy * (unsigned)nx), iy = (int)uy;
  MaxAbs wmax;
  for (int i = tid; i < 9 * MV * THS; i += NT) {
    const int r = i / (MV * THS), rem = i - r * (MV * THS);
    int cx = ix + r % 3 - 1, cy = iy + r / 3 - 1;
    cx += cx < 0 ? nx : (cx >= nx ? -nx : 0);
    cy += cy < 0 ? ny : (cy >= ny ? -ny : 0);
    const double q = Qg[((long long)cy * nx + cx) * (MV * THS) + rem];
    Qs[i] = q;
    wmax.add(q);
    const int j = rem / THS, s = rem - j * THS;
    double* w = Ws + (r * MV + j) * K::THT + s;  // Q^n extended constant in time
    w[0] = q;
#pragma unroll
    for (int t = 1; t < NB; ++t) w[t * THS] = 0.0;
  }
  int buf = 0;
  int whi = block_max_hi<NW>(wmax, red, buf);  // the iterate's largest entry, by its high word
  auto on_scale_of = [&](int ex) {             // and on a right-hand side's scale
    return ex >= -100 ? max_of_hi(whi) * scalbnf(1.f, -ex)
                      : (float)(__hiloint2double(whi, 0) * pow2(-ex));
  };

  // thread constants
  Rows<NB> R;
  {
    const int c = tid < COL ? tid : 0, r = c / THS, s = c - r * THS, y = s / NB, x = s - y * NB;
    const int ry = r / 3, rx = r - 3 * ry;
    const float l0 = keep((float)lam[0]), l1 = keep((float)lam[1]);
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      R.dx[n] = -l0 * T.D[x][n];
      R.dy[n] = -l1 * T.D[y][n];
    }
    R.xp = l0 * T.E[0][x];
    R.xm = -l0 * T.E[1][x];
    R.yp = l1 * T.E[0][y];
    R.ym = -l1 * T.E[1][y];
    R.gx = r * THS + y * NB;
    R.gy = r * THS + x;
    R.fx = (ry * 4 + rx) * VT * NB + y;
    R.fy = (12 + rx * 4 + ry) * VT * NB + x;
    const int f = tid < K::FL ? tid / NB : 0, o = tid < K::FL ? tid - f * NB : 0;
    int cl, cr;
    face_cells(f, R.dd, cl, cr);
    const int st = R.dd ? 1 : NB;
    R.bl = cl < 0 ? -1 : cl * THS + o * st;
    R.br = cr < 0 ? -1 : cr * THS + o * st;
  }
  Lin<NB, MV> S;
  const float g1 = keep((float)(a.gamma - 1.0));
  int it = 0;
  bool conv = false, capped = false, lin = true;
  float dprev = 0.f, bprev = 0.f;
  const int solves = F64 ? a.max_iters : min(kMaxSolves, a.max_solves);
#pragma unroll 1
  for (int solve = 0; solve < solves; ++solve) {
    if (solve == 0)
      residual<NB, MV, FLUX, true>(T, Ws, Qs, Rs, alpha, arena, lam, a.gamma);
    else
      residual<NB, MV, FLUX, false>(T, Ws, Qs, Rs, alpha, arena, lam, a.gamma);
    // exponent of the right-hand side (scaled by it, its squares stay normal in FP32)
    float rmax;
    int ex;
    if (!rhs_scale<NB, MV>(Rs, red, buf, rmax, ex)) break;
    float wrel = on_scale_of(ex);
    // mixed: a new linearisation where the last one no longer contracts by 3e3 per solve
    if (F64 || (solve > 0 && rmax > 3e-4f * bprev && it < a.max_iters)) lin = true;
    bprev = rmax;
    if (lin) {
      linearise<NB, MV>(T, Ws, R, S, P, g1);
      R.al = keep(0.5f * (float)alpha[tid < K::FL ? tid / NB : 0]);
      lin = F64;
      ++it;
    }
    // the update: its largest entry, rounded up so that the test below is never looser than
    // with FP64 maxima (the FP32 modes in P, unscaled by a power of two, are exact; FP64 ones are
    // known from their high words), and the iterate's, rounded down
    float ratio, dn;
    MaxAbs wm;
    if constexpr (!F64) {
      // relative accuracy: 1e-4 in the first solve (whose result the nonlinearity limits), then
      // down to an absolute ~1e-15 of the iterate, at most 1e-5 (FP32)
      const float rmin = solve == 0 ? 1e-4f : 1e-5f, rtop = solve == 0 ? 1e-4f : 1e-2f;
      if (!bicgstab<NB, MV, FLUX>(T, R, S, Rs, ex, 1e-15f * wrel, rmin, rtop, P, G, Fh, red, buf,
                                  g1, ratio))
        break;
      const double unscale = pow2(ex);
      float zm[1] = {0.f};
      for (int i = tid; i < 9 * BS; i += NT) {
        const float z = P[p_index<NB, MV>(i)];
        const double w = fma(-unscale, (double)z, Ws[i]);
        Ws[i] = w;
        zm[0] = fabsf(z) <= 1e30f ? fmaxf(zm[0], fabsf(z)) : 3e38f;  // (a NaN compares false)
        wm.add(w);
      }
      reduce<NW, 1, true>(zm, red, buf);
      dn = zm[0] <= 1e30f ? scalbnf(zm[0], ex) : 3e38f;
    } else {
      bool ok = true;
#pragma unroll 1
      for (int ref = 0;; ++ref) {
        if (ref > 0) {
          if (!rhs_scale<NB, MV>(Rs, red, buf, rmax, ex)) ok = false;
          wrel = on_scale_of(ex);
        }
        ok = ok && ref < kMaxRefine &&
             bicgstab<NB, MV, FLUX>(T, R, S, Rs, ex, 1e-17f * wrel, 3e-6f, 1e-3f, P, G, Fh, red,
                                    buf, g1, ratio);
        if (!ok) break;
        const double unscale = pow2(ex);
        float zm[1] = {0.f};
        for (int i = tid; i < 9 * BS; i += NT) {
          const float zf = P[p_index<NB, MV>(i)];
          const double z = unscale * (double)zf;
          Zs[i] = z;
          Ds[i] = ref == 0 ? z : Ds[i] + z;
          zm[0] = fabsf(zf) <= 1e30f ? fmaxf(zm[0], fabsf(zf)) : 3e38f;
        }
        reduce<NW, 1, true>(zm, red, buf);
        if (!(zm[0] <= 1e30f)) ok = false;
        // what is left of the linear system is below the iterate's round-off
        if (!ok || zm[0] * fmaxf(ratio, 1e-6f) <= 5e-17f * wrel) break;
        linear_update<NB, MV, FLUX>(TJ, T.Mt, Ws, Zs, Rs, alpha, arena, lam, a.gamma);
      }
      if (!ok) break;
      MaxAbs dm;
      for (int i = tid; i < 9 * BS; i += NT) {
        const double d = Ds[i], w = Ws[i] - d;
        Ws[i] = w;
        dm.add(d);
        wm.add(w);
      }
      ++dm.hi;  // rounded up
      dn = block_max<NW>(dm, red, buf) * 1.0000002f;
    }
    whi = block_max_hi<NW>(wm, red, buf);
    const float wn = max_of_hi(whi);
    if (!(dn < 1e30f) || !(wn < 1e30f)) break;
    if ((double)dn <= a.tol * fmax(1.0, (double)wn)) {
      conv = true;
      break;
    }
    if (!F64 && solve > 0 && dn > 0.1f * dprev) break;
    dprev = dn;
    // the FP64 iterates are the block elimination's to round-off, also at the cap (a tolerance
    // below round-off, where the two differ, stays the block elimination's to decide)
    capped = F64 && solve + 1 == solves && (double)dn > 1e-12 * fmax(1.0, (double)wn);
  }
  if (conv || capped) {
    for (int i = tid; i < BS; i += NT) Wg[e * BS + i] = Ws[4 * BS + i];
    if (tid == 0) {
      if (!conv) atomicAdd(&stats[0], 1);
      atomicMax(&stats[1], it);
      atomicAdd(&stats[7 + (it < 15 ? it : 15)], 1);
      atomicAdd(itot, (unsigned long long)it);
    }
  } else if (tid == 0) {
    a.list[atomicAdd(a.list_count, 1)] = (int)eg;
  }
}

}  // namespace mf
}  // namespace ridg
