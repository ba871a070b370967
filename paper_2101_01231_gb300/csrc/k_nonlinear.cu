// Nonlinear flux in 2D: host tables on the device, the block elimination plan of the
// 3 x 3 region Jacobian, the correction step (Sec. 2.3) with quadrature, and the wave-speed
// reduction that sets dt.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "k_nl_lines.cuh"
#include "nl_tables.h"
#include "ridg_internal.h"
#include "tables.h"

namespace ridg {

// ---------------------------------------------------------------------------------------
// tables
// ---------------------------------------------------------------------------------------
int nl_tables_upload(int nb, NlDevTables& out, void* mem, size_t* bytes, cudaStream_t s) {
  NlHostTables t = build_nl_tables(nb - 1);
  // 6 x 6 equispaced points of the wave-speed estimate
  std::vector<double> eq(6);
  for (int i = 0; i < 6; ++i) eq[i] = -1.0 + 2.0 * i / 5.0;
  std::vector<double> phieq((size_t)t.thS * 36);
  {
    std::vector<double> v(nb), dv(nb);
    std::vector<double> V((size_t)nb * 6);
    for (int i = 0; i < 6; ++i) {
      phi_values(nb, eq[i], v.data(), dv.data());
      for (int b = 0; b < nb; ++b) V[(size_t)b * 6 + i] = v[b];
    }
    for (int s2 = 0; s2 < t.thS; ++s2)
      for (int iy = 0; iy < 6; ++iy)
        for (int ix = 0; ix < 6; ++ix)
          phieq[(size_t)s2 * 36 + iy * 6 + ix] = V[(size_t)(s2 % nb) * 6 + ix] * V[(size_t)(s2 / nb) * 6 + iy];
  }
  struct Piece {
    const void* src;
    size_t n;
    size_t off;
  };
  std::vector<Piece> pieces;
  size_t off = 0;
  auto add = [&](const void* src, size_t nbytes) {
    off = (off + 255) & ~(size_t)255;
    pieces.push_back({src, nbytes, off});
    off += nbytes;
    return pieces.size() - 1;
  };
  auto addd = [&](const std::vector<double>& v) { return add(v.data(), v.size() * sizeof(double)); };
  auto addi = [&](const std::vector<int>& v) { return add(v.data(), v.size() * sizeof(int)); };
  const size_t iMt = addd(t.Mt), iem = addd(t.em), iwV = addd(t.wV), iPsiF = addd(t.PsiF), iwF = addd(t.wF), iPsiAtP = addd(t.PsiAtP),
               iPsiAtFP = addd(t.PsiAtFP), iP1 = addd(t.P1), iPhiEq = addd(phieq);
  const size_t iV1 = addd(t.V1), iV1T = addd(t.V1T), idV1 = addd(t.dV1), iep1 = addd(t.ep1),
               iem1 = addd(t.em1);
  // merged assembly lists, packed per precision
  NlAsmLists L = build_asm_lists(t);
  struct EntD { int off; int pad; double c; };
  struct EntF { int off; float c; };
  auto packd = [](const std::vector<int>& o, const std::vector<double>& v) {
    std::vector<EntD> e(o.size());
    for (size_t i = 0; i < o.size(); ++i) e[i] = {o[i], 0, v[i]};
    return e;
  };
  auto packf = [](const std::vector<int>& o, const std::vector<double>& v) {
    std::vector<EntF> e(o.size());
    for (size_t i = 0; i < o.size(); ++i) e[i] = {o[i], (float)v[i]};
    return e;
  };
  std::vector<EntD> dd_ = packd(L.doff, L.dval);
  std::vector<EntF> df_ = packf(L.doff, L.dval);
  std::vector<EntD> od_[4];
  std::vector<EntF> of_[4];
  for (int f = 0; f < 4; ++f) {
    od_[f] = packd(L.ooff[f], L.oval[f]);
    of_[f] = packf(L.ooff[f], L.oval[f]);
  }
  const size_t idptr = addi(L.dptr), identd = add(dd_.data(), dd_.size() * sizeof(EntD)),
               identf = add(df_.data(), df_.size() * sizeof(EntF));
  size_t ioptr[4], ioentd[4], ioentf[4];
  for (int f = 0; f < 4; ++f) {
    ioptr[f] = addi(L.optr[f]);
    ioentd[f] = add(od_[f].data(), od_[f].size() * sizeof(EntD));
    ioentf[f] = add(of_[f].data(), of_[f].size() * sizeof(EntF));
  }
  auto tof = [](const std::vector<double>& v) { return std::vector<float>(v.begin(), v.end()); };
  std::vector<float> Mtf = tof(t.Mt), PsiAtPf = tof(t.PsiAtP), PsiAtFPf = tof(t.PsiAtFP), P1f = tof(t.P1);
  std::vector<float> T0f = tof(t.T0), T1f = tof(t.T1), ep1f = tof(t.ep1), em1f = tof(t.em1);
  const size_t iMtf = add(Mtf.data(), Mtf.size() * 4), iPsiAtPf = add(PsiAtPf.data(), PsiAtPf.size() * 4),
               iPsiAtFPf = add(PsiAtFPf.data(), PsiAtFPf.size() * 4), iP1f = add(P1f.data(), P1f.size() * 4);
  const size_t iT0f = add(T0f.data(), T0f.size() * 4), iT1f = add(T1f.data(), T1f.size() * 4),
               iep1f = add(ep1f.data(), ep1f.size() * 4), iem1f = add(em1f.data(), em1f.size() * 4);
  const size_t total = (off + 255) & ~(size_t)255;
  if (!mem) {
    *bytes = total;
    return RIDG_OK;
  }
  if (*bytes < total) return RIDG_EINVAL;
  char* base = (char*)mem;
  for (const Piece& p : pieces)
    if (p.n && cudaMemcpyAsync(base + p.off, p.src, p.n, cudaMemcpyHostToDevice, s) != cudaSuccess)
      return RIDG_ECUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return RIDG_ECUDA;  // host vectors go away
  auto D = [&](size_t i) { return (const double*)(base + pieces[i].off); };
  auto I = [&](size_t i) { return (const int*)(base + pieces[i].off); };
  NlDev& tb = out.tb;
  tb.Mt = D(iMt);
  tb.em = D(iem);
  tb.wV = D(iwV);
  tb.PsiF = D(iPsiF);
  tb.wF = D(iwF);
  tb.PsiAtP = D(iPsiAtP);
  tb.PsiAtFP = D(iPsiAtFP);
  tb.P1 = D(iP1);
  tb.PhiEq = D(iPhiEq);
  tb.V1 = D(iV1);
  tb.V1T = D(iV1T);
  tb.dV1 = D(idV1);
  tb.ep1 = D(iep1);
  tb.em1 = D(iem1);
  tb.dptr = I(idptr);
  tb.dent_d = base + pieces[identd].off;
  tb.dent_f = base + pieces[identf].off;
  for (int f = 0; f < 4; ++f) {
    tb.optr[f] = I(ioptr[f]);
    tb.oent_d[f] = base + pieces[ioentd[f]].off;
    tb.oent_f[f] = base + pieces[ioentf[f]].off;
  }
  auto F = [&](size_t i) { return (const float*)(base + pieces[i].off); };
  tb.Mt_f = F(iMtf);
  tb.PsiAtP_f = F(iPsiAtPf);
  tb.PsiAtFP_f = F(iPsiAtFPf);
  tb.P1_f = F(iP1f);
  tb.T0_f = F(iT0f);
  tb.T1_f = F(iT1f);
  tb.ep1_f = F(iep1f);
  tb.em1_f = F(iem1f);
  out.mem = mem;
  out.bytes = total;
  return RIDG_OK;
}

namespace {

// ---------------------------------------------------------------------------------------
// correction (Sec. 2.3): Q += volume term - surface term, every face flux evaluated from the
// same traces in the same order by both cells that share it (so both see the same bits)
//
// Sum-factorised along lines (k_nl_lines.cuh): a cell takes ~9 k FP64 operations at Burgers Q4
// where sums over the dense quadrature tables took ~95 k.  The FP64 pipe bounds it; a block
// takes CPB cells so that its phases of 16 to 50 lines per cell fill their warps.  Measured:
// Euler Q2 512^2 21.2 -> 7.8 ms per launch; eight Burgers problems up to 72^2, degrees 1 .. 4,
// 13.2 -> 10.8 ms per whole step.
// ---------------------------------------------------------------------------------------
constexpr int kCorrThreads = 128;

template <int NB, int MV>
struct CorrCfg {
  static constexpr int THS = NB * NB, BS = MV * NB * THS, NQ = nl::Rule<NB>::NQ, NX = NQ * NQ;
  // cells per block: about 128 points of the volume phase (NQ^2 per cell)
  static constexpr int CPB = NB == 2 ? (MV == 1 ? 16 : 8) : NB == 3 ? (MV == 1 ? 8 : 4) : NB == 4 ? 5 : 3;
  // shared memory of a cell (doubles): lines [j][a][y][x]; traces [face * 2 + left / right][j][a]
  // [NQ]; time-summed fluxes [x, y][j][y][x]; speeds [face][NQ]; face values [face][j][NQ]
  static constexpr int oT = MV * NB * NX, oG = oT + 8 * MV * NB * NQ, oS = oG + 2 * MV * NX,
                       oH = oS + 4 * NQ, per_cell = oH + 4 * MV * NQ, total = CPB * per_cell;
};

// The correction of cells e0 .. min(e0 + CPB, end) - 1 of one mesh by the block.  Faces of a
// cell: f = dd * 2 + si (si 0: the +1 face, 1: the -1 face) with left / right states
//   +1 face: own trace at +1, the +dd neighbour's at -1;
//   -1 face: the -dd neighbour's at +1, own at -1.
template <int NB, int MV, int FLUX>
__device__ void nl_correct_cells(const nl::Rule<NB>& T, double* __restrict__ Q,
                                 const double* __restrict__ W, int nx, int ny, long long end,
                                 double lamx, double lamy, double g, long long e0, double* sh) {
  using K = CorrCfg<NB, MV>;
  constexpr int NQ = K::NQ, NX = K::NX, THS = K::THS, BS = K::BS, ML = MV * NB;
  const int tid = threadIdx.x;
  const int cells = (int)min((long long)K::CPB, end - e0);
  // x lines of the cell and its x traces | its y traces | the neighbours' traces per face
  for (int i = tid; i < cells * 6 * ML * NB; i += kCorrThreads) {
    const int c = i / (6 * ML * NB), k = i - c * (6 * ML * NB), kind = k / (ML * NB),
              l = k - kind * (ML * NB), ja = l / NB, o = l - ja * NB;
    double* S = sh + c * K::per_cell;
    double* tr = S + K::oT + ja * NQ + o;  // + (face * 2 + side) ML NQ
    const long long e = e0 + c;
    const unsigned uy = (unsigned)e / (unsigned)nx;
    int cx = (int)((unsigned)e - uy * (unsigned)nx), cy = (int)uy;
    if (kind >= 2) {
      const int f = kind - 2, step = (f & 1) ? -1 : 1;
      if (f < 2) cx += step; else cy += step;
      cx += cx < 0 ? nx : (cx >= nx ? -nx : 0);
      cy += cy < 0 ? ny : (cy >= ny ? -ny : 0);
    }
    const double* src = W + ((long long)cy * nx + cx) * BS + ja * THS;
    const bool ydir = kind == 1 || kind >= 4;
    const int st = ydir ? NB : 1;
    src += ydir ? o : o * NB;
    double m[NB], ev, od;
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = src[b * st];
    nl::traces(T, m, 1, ev, od);
    if (kind == 0) {
      double v[NQ];
      nl::interp(T, m, v);
#pragma unroll
      for (int q = 0; q < NQ; ++q) S[(ja * NQ + o) * NQ + q] = v[q];
    }
    if (kind < 2) {
      tr[(kind * 4 + 0) * ML * NQ] = ev + od;  // left of the +1 face
      tr[(kind * 4 + 3) * ML * NQ] = ev - od;  // right of the -1 face
    } else {
      const int f = kind - 2;  // right of the +1 faces, left of the -1 faces
      tr[(f * 2 + ((f & 1) ? 0 : 1)) * ML * NQ] = (f & 1) ? ev + od : ev - od;
    }
  }
  __syncthreads();
  // y lines; the traces along their faces
  for (int i = tid; i < cells * (ML * NQ + 8 * ML); i += kCorrThreads) {
    const int c = i / (ML * NQ + 8 * ML), k = i - c * (ML * NQ + 8 * ML);
    double* p = sh + c * K::per_cell;
    int st = 1;
    if (k < ML * NQ) {
      p += k / NQ * NX + k % NQ;
      st = NQ;
    } else {
      p += K::oT + (k - ML * NQ) * NQ;
    }
    double m[NB], v[NQ];
#pragma unroll
    for (int b = 0; b < NB; ++b) m[b] = p[b * st];
    nl::interp(T, m, v);
#pragma unroll
    for (int q = 0; q < NQ; ++q) p[q * st] = v[q];
  }
  __syncthreads();
  // volume points: both fluxes summed over time; face points: the largest speed over time
  for (int i = tid; i < cells * NX; i += kCorrThreads) {
    const int c = i / NX, yx = i - c * NX;
    double* S = sh + c * K::per_cell;
    double sx[MV], sy[MV];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double w[MV], fx[MV], fy[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        w[j] = S[j * NB * NX + yx];
#pragma unroll
        for (int a = 1; a < NB; ++a) w[j] = fma(nl::vq(T, a, q), S[(j * NB + a) * NX + yx], w[j]);
      }
      nl::flux2<FLUX, true>(w, fx, fy, g);
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        const double wt = nl::wvq(T, 0, q);
        sx[j] = q == 0 ? wt * fx[j] : fma(wt, fx[j], sx[j]);
        if constexpr (MV > 1) sy[j] = q == 0 ? wt * fy[j] : fma(wt, fy[j], sy[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < MV; ++j) {
      S[K::oG + j * NX + yx] = sx[j];
      if constexpr (MV > 1) S[K::oG + (MV + j) * NX + yx] = sy[j];
    }
  }
  for (int i = tid; i < cells * 4 * NQ; i += kCorrThreads) {
    const int c = i / (4 * NQ), k = i - c * (4 * NQ), f = k / NQ, qo = k - f * NQ, dd = f >> 1;
    double* S = sh + c * K::per_cell;
    const double* tl = S + K::oT + f * 2 * ML * NQ + qo;
    const double* tr = tl + ML * NQ;
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double wl[MV], wr[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        wl[j] = tl[j * NB * NQ];
        wr[j] = tr[j * NB * NQ];
#pragma unroll
        for (int a = 1; a < NB; ++a) {
          wl[j] = fma(nl::vq(T, a, q), tl[(j * NB + a) * NQ], wl[j]);
          wr[j] = fma(nl::vq(T, a, q), tr[(j * NB + a) * NQ], wr[j]);
        }
      }
      s = fmax(s, fmax(nlflux::speed<FLUX>(wl, dd, g), nlflux::speed<FLUX>(wr, dd, g)));
    }
    S[K::oS + k] = s;
  }
  __syncthreads();
  // the face fluxes summed over time; the volume fluxes' y lines back (phi_y on the x flux,
  // phi_y' on the y flux)
  for (int i = tid; i < cells * 4 * NQ; i += kCorrThreads) {
    const int c = i / (4 * NQ), k = i - c * (4 * NQ), f = k / NQ, qo = k - f * NQ, dd = f >> 1;
    double* S = sh + c * K::per_cell;
    const double* tl = S + K::oT + f * 2 * ML * NQ + qo;
    const double* tr = tl + ML * NQ;
    double alpha = 0.0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) alpha = fmax(alpha, S[K::oS + f * NQ + q]);
    alpha *= 0.5;
    double h[MV];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double wl[MV], wr[MV], fl[MV], fr[MV];
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        wl[j] = tl[j * NB * NQ];
        wr[j] = tr[j * NB * NQ];
#pragma unroll
        for (int a = 1; a < NB; ++a) {
          wl[j] = fma(nl::vq(T, a, q), tl[(j * NB + a) * NQ], wl[j]);
          wr[j] = fma(nl::vq(T, a, q), tr[(j * NB + a) * NQ], wr[j]);
        }
      }
      nl::flux1<FLUX, true>(wl, dd, fl, g);
      nl::flux1<FLUX, true>(wr, dd, fr, g);
#pragma unroll
      for (int j = 0; j < MV; ++j) {
        const double fh = fma(0.5, fl[j] + fr[j], -alpha * (wr[j] - wl[j]));
        const double wt = nl::wvq(T, 0, q);
        h[j] = q == 0 ? wt * fh : fma(wt, fh, h[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < MV; ++j) S[K::oH + (f * MV + j) * NQ + qo] = h[j];
  }
  for (int i = tid; i < cells * MV * NQ; i += kCorrThreads) {
    const int c = i / (MV * NQ), k = i - c * (MV * NQ), j = k / NQ, x = k - j * NQ;
    double* p1 = sh + c * K::per_cell + K::oG + j * NX + x;
    double* p2 = p1 + MV * NX;
    double v[NQ], o1[NB], o2[NB];
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = p1[q * NQ];
    nl::project<false>(T, v, o1);
    if constexpr (MV > 1) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = p2[q * NQ];
    }
    nl::project<true>(T, v, o2);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      p1[b * NQ] = o1[b];
      p2[b * NQ] = o2[b];
    }
  }
  __syncthreads();
  for (int i = tid; i < cells * 4 * MV; i += kCorrThreads) {
    double* p = sh + i / (4 * MV) * K::per_cell + K::oH + i % (4 * MV) * NQ;
    double v[NQ], o[NB];
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = p[q];
    nl::project<false>(T, v, o);
#pragma unroll
    for (int b = 0; b < NB; ++b) p[b] = o[b];
  }
  __syncthreads();
  // x lines back, the faces, and the update
  const double l0 = 0.25 * lamx, l1 = 0.25 * lamy;
  for (int i = tid; i < cells * MV * NB; i += kCorrThreads) {
    const int c = i / (MV * NB), k = i - c * (MV * NB), j = k / NB, y = k - j * NB;
    const double* S = sh + c * K::per_cell;
    const double* p1 = S + K::oG + j * NX + y * NQ;
    double v[NQ], ox[NB], oy[NB];
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = p1[q];
    nl::project<true>(T, v, ox);
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = p1[MV * NX + q];
    nl::project<false>(T, v, oy);
    const double* h = S + K::oH + j * NQ;  // + face MV NQ
    const double hr = h[y], hl = h[MV * NQ + y];
    double* q = Q + ((e0 + c) * MV + j) * THS + y * NB;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const double ht = h[2 * MV * NQ + b], hb = h[3 * MV * NQ + b];
      const double fx = (b & 1) ? hr + hl : hr - hl, fy = (y & 1) ? ht + hb : ht - hb;
      const double d = fma(l0, fma(-T.ep[b], fx, ox[b]), l1 * fma(-T.ep[y], fy, oy[b]));
      q[b] += d;
    }
  }
}

template <int NB, int MV, int FLUX>
__global__ void __launch_bounds__(kCorrThreads) nl_correct_kernel(const nl::Rule<NB> T,
                                                                  double* __restrict__ Q,
                                                                  const double* __restrict__ W,
                                                                  int nx, int ny, long long ncell,
                                                                  double lamx, double lamy,
                                                                  double gamma, int cpb) {
  __shared__ double sh[CorrCfg<NB, MV>::total];
  const long long e0 = (long long)blockIdx.x * cpb;
  nl_correct_cells<NB, MV, FLUX>(T, Q, W, nx, ny, min(ncell, e0 + cpb), lamx, lamy, gamma, e0, sh);
}

struct CorrRules {
  nl::Rule<2> r2;
  nl::Rule<3> r3;
  nl::Rule<4> r4;
  nl::Rule<5> r5;
};

// Every instance's correction of a batched Burgers ensemble in one launch: each instance has
// ceil(ncell / CPB) blocks of its degree, the instance of a block found by bisection.
__global__ void __launch_bounds__(kCorrThreads) nl_correct_multi_kernel(const CorrMulti m,
                                                                        const CorrRules T) {
  __shared__ double sh[std::max(std::max(CorrCfg<2, 1>::total, CorrCfg<3, 1>::total),
                                std::max(CorrCfg<4, 1>::total, CorrCfg<5, 1>::total))];
  const long long b = blockIdx.x;
  int lo = 0, hi = m.ninst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (m.inst[mid].block0 <= b) lo = mid; else hi = mid - 1;
  }
  const CorrInst& in = m.inst[lo];
  const long long k = b - in.block0;
  switch (in.nb) {
    case 2: nl_correct_cells<2, 1, RIDG_FLUX_BURGERS>(T.r2, in.Q, in.W, in.nx, in.ny, in.ncell, in.lamx, in.lamy, 0.0, k * CorrCfg<2, 1>::CPB, sh); break;
    case 3: nl_correct_cells<3, 1, RIDG_FLUX_BURGERS>(T.r3, in.Q, in.W, in.nx, in.ny, in.ncell, in.lamx, in.lamy, 0.0, k * CorrCfg<3, 1>::CPB, sh); break;
    case 4: nl_correct_cells<4, 1, RIDG_FLUX_BURGERS>(T.r4, in.Q, in.W, in.nx, in.ny, in.ncell, in.lamx, in.lamy, 0.0, k * CorrCfg<4, 1>::CPB, sh); break;
    case 5: nl_correct_cells<5, 1, RIDG_FLUX_BURGERS>(T.r5, in.Q, in.W, in.nx, in.ny, in.ncell, in.lamx, in.lamy, 0.0, k * CorrCfg<5, 1>::CPB, sh); break;
    default: break;
  }
}

template <int NB, int MV, int FLUX>
__global__ void max_speed_kernel(NlDev tb, const double* __restrict__ Q, long long ncell,
                                 double gamma, unsigned long long* out) {
  constexpr int THS = NB * NB;
  double best = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < ncell * 36;
       i += (long long)gridDim.x * blockDim.x) {
    const long long e = i / 36;
    const int pnt = (int)(i % 36);
    double w[MV];
    for (int j = 0; j < MV; ++j) {
      double acc = 0.0;
      for (int s2 = 0; s2 < THS; ++s2) acc = fma(tb.PhiEq[s2 * 36 + pnt], Q[(e * MV + j) * THS + s2], acc);
      w[j] = acc;
    }
    for (int dd = 0; dd < 2; ++dd) best = fmax(best, nlflux::speed<FLUX>(w, dd, gamma));
  }
  for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
  // speeds are >= 0, so their bit patterns order like their values (a NaN state is refused
  // by the finite check before this runs)
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(best));
}

}  // namespace

#define RIDG_NL_SWITCH(NB_, M_, KIND_, ...)                                               \
  do {                                                                                    \
    if (KIND_ == RIDG_FLUX_BURGERS && M_ == 1) {                                          \
      switch (NB_) {                                                                      \
        case 2: { constexpr int NB = 2, MV = 1, FL = RIDG_FLUX_BURGERS; __VA_ARGS__; } break;    \
        case 3: { constexpr int NB = 3, MV = 1, FL = RIDG_FLUX_BURGERS; __VA_ARGS__; } break;    \
        case 4: { constexpr int NB = 4, MV = 1, FL = RIDG_FLUX_BURGERS; __VA_ARGS__; } break;    \
        case 5: { constexpr int NB = 5, MV = 1, FL = RIDG_FLUX_BURGERS; __VA_ARGS__; } break;    \
        default: return cudaErrorInvalidValue;                                            \
      }                                                                                   \
    } else if (KIND_ == RIDG_FLUX_EULER && M_ == 4) {                                     \
      switch (NB_) {                                                                      \
        case 2: { constexpr int NB = 2, MV = 4, FL = RIDG_FLUX_EULER; __VA_ARGS__; } break;      \
        case 3: { constexpr int NB = 3, MV = 4, FL = RIDG_FLUX_EULER; __VA_ARGS__; } break;      \
        default: return cudaErrorInvalidValue;                                            \
      }                                                                                   \
    } else {                                                                              \
      return cudaErrorInvalidValue;                                                       \
    }                                                                                     \
  } while (0)

cudaError_t launch_newton_f64(int nb, int m, int kind, const NewtonArgs& a, int grid,
                              cudaStream_t s);
cudaError_t launch_newton_f32(int nb, int m, int kind, const NewtonArgs& a, int grid,
                              cudaStream_t s);
cudaError_t launch_newton_tf32(int nb, int m, int kind, const NewtonArgs& a, int grid,
                               cudaStream_t s);

bool newton_supported(int nb, int m) { return (m == 1 && nb >= 2 && nb <= 5) || (m == 4 && nb >= 2 && nb <= 3); }

int newton_ctas_per_sm_f64(int nb, int m, int kind);
int newton_ctas_per_sm_f32(int nb, int m, int kind);
int newton_ctas_per_sm_tf32(int nb, int m, int kind);

int newton_grid(int nb, int m, int kind, int prec) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return 0;
  const int per = prec == kNewtonTF32  ? newton_ctas_per_sm_tf32(nb, m, kind)
                  : prec == kNewtonF32 ? newton_ctas_per_sm_f32(nb, m, kind)
                                       : newton_ctas_per_sm_f64(nb, m, kind);
  return per > 0 ? per * sms : 0;  // a persistent grid: every resident CTA slot filled once
}

size_t newton_scratch_per_cta(int nb, int m, int prec, const NlPlan& plan) {
  const int bs = m * nb * nb * nb, bp = (bs + 15) / 16 * 16;
  const size_t bytes =
      (size_t)plan.nslots * bp * bp * (prec == kNewtonF64 ? sizeof(double) : sizeof(float));
  return (bytes + 255) & ~(size_t)255;
}

cudaError_t launch_newton(int nb, int m, int flux_kind, int prec, const NewtonArgs& a, int grid,
                          cudaStream_t s) {
  switch (prec) {
    case kNewtonF64: return launch_newton_f64(nb, m, flux_kind, a, grid, s);
    case kNewtonF32: return launch_newton_f32(nb, m, flux_kind, a, grid, s);
    case kNewtonTF32: return launch_newton_tf32(nb, m, flux_kind, a, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_newton_multi_f64(const NewtonMulti& m, const NewtonMulti* dev, int grid,
                                 cudaStream_t s);
cudaError_t launch_newton_multi_f32(const NewtonMulti& m, const NewtonMulti* dev, int grid,
                                 cudaStream_t s);
cudaError_t launch_newton_multi_tf32(const NewtonMulti& m, const NewtonMulti* dev, int grid,
                                 cudaStream_t s);
int newton_multi_ctas_per_sm_f64();
int newton_multi_ctas_per_sm_f32();
int newton_multi_ctas_per_sm_tf32();

cudaError_t launch_newton_multi(int prec, const NewtonMulti& m, const NewtonMulti* dev, int grid,
                                cudaStream_t s) {
  switch (prec) {
    case kNewtonF64: return launch_newton_multi_f64(m, dev, grid, s);
    case kNewtonF32: return launch_newton_multi_f32(m, dev, grid, s);
    case kNewtonTF32: return launch_newton_multi_tf32(m, dev, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

int newton_multi_ctas_per_sm(int prec) {
  switch (prec) {
    case kNewtonF64: return newton_multi_ctas_per_sm_f64();
    case kNewtonF32: return newton_multi_ctas_per_sm_f32();
    case kNewtonTF32: return newton_multi_ctas_per_sm_tf32();
    default: return 0;
  }
}

cudaError_t launch_nl_correct(int nb, int m, int flux_kind, double* Q, const double* W, int nx,
                              int ny, long long ncell, double lamx, double lamy, double gamma,
                              cudaStream_t s) {
  RIDG_NL_SWITCH(nb, m, flux_kind, {
    // fewer cells per block where that leaves SMs without one (3 x 3 cells, Euler Q1, 22.5 -> 20.5 us)
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int cpb = (int)std::min<long long>(CorrCfg<NB, MV>::CPB, (ncell + sms - 1) / sms);
    static const nl::Rule<NB> rule = nl::make_rule<NB>();
    (nl_correct_kernel<NB, MV, FL><<<(unsigned)((ncell + cpb - 1) / cpb), kCorrThreads, 0, s>>>(
        rule, Q, W, nx, ny, ncell, lamx, lamy, gamma, cpb));
  });
  return cudaGetLastError();
}

long long nl_correct_blocks(int nb, long long ncell) {
  const int cpb = nb == 2   ? CorrCfg<2, 1>::CPB
                  : nb == 3 ? CorrCfg<3, 1>::CPB
                  : nb == 4 ? CorrCfg<4, 1>::CPB
                            : CorrCfg<5, 1>::CPB;
  return (ncell + cpb - 1) / cpb;
}

cudaError_t launch_nl_correct_multi(const CorrMulti& m, long long blocks, cudaStream_t s) {
  static const CorrRules rules = {nl::make_rule<2>(), nl::make_rule<3>(), nl::make_rule<4>(),
                                  nl::make_rule<5>()};
  nl_correct_multi_kernel<<<(unsigned)blocks, kCorrThreads, 0, s>>>(m, rules);
  return cudaGetLastError();
}

cudaError_t launch_max_speed(int nb, int m, int flux_kind, const NlDev& tb, const double* Q,
                             long long ncell, double gamma, unsigned long long* out,
                             cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  const long long work = ncell * 36;
  const unsigned blocks = (unsigned)std::min<long long>((work + 255) / 256, 4096);
  RIDG_NL_SWITCH(nb, m, flux_kind,
                 (max_speed_kernel<NB, MV, FL><<<blocks, 256, 0, s>>>(tb, Q, ncell, gamma, out)));
  return cudaGetLastError();
}

}  // namespace ridg
