// FP64 kernels of the linear-flux RIDG step.
//
// Prediction (Sec. 2.2): for a linear flux on a uniform periodic mesh the region system
// of eq. pred_full_system is the same for every cell, so the kept centre coefficients
// are W_i = P X_i with X_i the theta_S coefficients of the region cells upstream of cell i
// (the upwind box, 2^d of the 3^d cells for a velocity with no zero component; the others
// have zero columns) gathered with periodic wrap, and P the centre rows of the region
// solution operator.
//
// Correction (Sec. 2.3): with W-bar the time mean of W (all a linear flux needs, since
// int psi_g dtau = 2 delta_g0),
//   dQ_i = sum_d nu_d (D along d) Wbar_i
//          - sum_d [ phi(+1) (x)_d F_{i+1/2} - phi(-1) (x)_d F_{i-1/2} ],
//   F_{i+1/2} = nu+_d trace_{+1}(Wbar_i) + nu-_d trace_{-1}(Wbar_{i+e_d}).
// Each face value is evaluated by one device function with a fixed fma order from the
// same inputs on both sides of the face, so the two neighbours apply bitwise the same
// flux and the cell averages are conserved to round-off of the final additions.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>

#include "k_pdl.cuh"
#include "ridg_internal.h"

namespace ridg {
namespace {

constexpr int ipow_c(int b, int e) { return e == 0 ? 1 : b * ipow_c(b, e - 1); }

struct Coords {
  int x, y, z;
};

// (cell counts stay below 2^31: 32-bit division, far cheaper than 64-bit)
__device__ __forceinline__ Coords cell_coords(long long e, int nx, int ny) {
  Coords c;
  const unsigned u = (unsigned)e, r = u / (unsigned)nx;
  c.x = (int)(u - r * (unsigned)nx);
  c.y = (int)(r % (unsigned)ny);
  c.z = (int)(r / (unsigned)ny);
  return c;
}

__device__ __forceinline__ int wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <int DIM>
__device__ __forceinline__ long long neighbour(const Coords& c, int ox, int oy, int oz, int nx,
                                               int ny, int nz) {
  long long j = wrap(c.x + ox, nx);
  if (DIM > 1) j += (long long)nx * wrap(c.y + oy, ny);
  if (DIM > 2) j += (long long)nx * ny * wrap(c.z + oz, nz);
  return j;
}

// ---------------------------------------------------------------------------------------
// prediction: each thread owns one cell and CH consecutive output rows of P
// ---------------------------------------------------------------------------------------
template <int DIM, int NB, int CH>
__global__ void __launch_bounds__(128) predict_fp64_kernel(const double* Q,
                                                           const double* __restrict__ P, int nout,
                                                           double* __restrict__ W, int wstride,
                                                           int nx, int ny, int nz, long long ncell,
                                                           RegionBox box) {
  constexpr int THS = ipow_c(NB, DIM);
  const int K = box.n * THS;
  extern __shared__ double sP[];  // CH x K
  const int c0 = blockIdx.y * CH;
  const int have = min(CH, nout - c0) * K;  // (the last rows may be padding)
#pragma unroll 8
  for (int i = threadIdx.x; i < CH * K; i += blockDim.x)
    sP[i] = i < have ? P[(size_t)c0 * K + i] : 0.0;
  grid_wait();
  __syncthreads();
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ncell) return;
  const Coords c = cell_coords(e, nx, ny);
  double acc[CH];
#pragma unroll
  for (int j = 0; j < CH; ++j) acc[j] = 0.0;
#pragma unroll 1
  for (int r = 0; r < box.n; ++r) {
    const int ox = box.lo[0] + r % box.cnt[0];
    const int oy = box.lo[1] + (r / box.cnt[0]) % box.cnt[1];
    const int oz = box.lo[2] + r / (box.cnt[0] * box.cnt[1]);
    const double* q = Q + neighbour<DIM>(c, ox, oy, oz, nx, ny, nz) * THS;
    const double* p = sP + r * THS;
#pragma unroll
    for (int s = 0; s < THS; ++s) {
      const double x = q[s];
#pragma unroll
      for (int j = 0; j < CH; ++j) acc[j] = fma(p[j * K + s], x, acc[j]);
    }
  }
  double* w = W + e * wstride + c0;
#pragma unroll
  for (int j = 0; j < CH; ++j)
    if (c0 + j < nout) w[j] = acc[j];
}

// ---------------------------------------------------------------------------------------
// correction
// ---------------------------------------------------------------------------------------
// The value of a face from the upwind cell's trace there: nu_d^+ tr_+(left) for nu_d > 0, nu_d^-
// tr_-(right) for nu_d < 0 (the other side's coefficient is zero), one product of one sum in a
// fixed order, so both neighbours evaluate it bit-identically.
struct Upwind {
  double nf;        // nu_d
  const double* v;  // phi_b(+1) or phi_b(-1)
  int up;           // offset of the upstream cell along d (0: no flux along d)
};
__device__ __forceinline__ Upwind upwind_of(const CorrParams& cp, int dd) {
  return cp.nu[dd] > 0.0 ? Upwind{cp.nu[dd], cp.ep, -1}
                         : Upwind{cp.nu[dd], cp.em, cp.nu[dd] < 0.0 ? 1 : 0};
}

// One thread per cell: the time means of the cell and of its upstream neighbour per direction.
template <int DIM, int NB>
__global__ void __launch_bounds__(128) correct_linear_kernel(double* Q, const double* Wb,
                                                             int wstride, int nx, int ny, int nz,
                                                             long long ncell, CorrParams cp) {
  constexpr int THS = ipow_c(NB, DIM);
  constexpr int NT = ipow_c(NB, DIM - 1);
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  grid_wait();
  if (e >= ncell) return;
  const Coords c = cell_coords(e, nx, ny);
  double w[THS], dq[THS];
#pragma unroll
  for (int s = 0; s < THS; ++s) {
    w[s] = Wb[e * wstride + s];
    dq[s] = 0.0;
  }
#pragma unroll
  for (int dd = 0; dd < DIM; ++dd) {
    const int st = dd == 0 ? 1 : (dd == 1 ? NB : NB * NB);
    const Upwind uw = upwind_of(cp, dd);
    const double* wu = Wb + neighbour<DIM>(c, dd == 0 ? uw.up : 0, dd == 1 ? uw.up : 0,
                                           dd == 2 ? uw.up : 0, nx, ny, nz) * wstride;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int base = t % st + (t / st) * st * NB;
      // volume term nu_d (D along d) Wbar
#pragma unroll
      for (int a = 0; a < NB; ++a) {
        double acc = 0.0;
#pragma unroll
        for (int b = 0; b < NB; ++b)
          if (a > b && ((a + b) & 1)) acc = fma(cp.D[a * kMaxNB + b], w[base + b * st], acc);
        dq[base + a * st] = fma(cp.nu[dd], acc, dq[base + a * st]);
      }
      double to = 0.0, tu = 0.0;
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        to = fma(uw.v[b], w[base + b * st], to);
        tu = fma(uw.v[b], wu[base + b * st], tu);
      }
      const double fo = uw.nf * to, fu = uw.nf * tu;
      const double fp = uw.up > 0 ? fu : fo, fm = uw.up > 0 ? fo : fu;
#pragma unroll
      for (int a = 0; a < NB; ++a) {
        double v = dq[base + a * st];
        v = fma(-cp.ep[a], fp, v);
        v = fma(cp.em[a], fm, v);
        dq[base + a * st] = v;
      }
    }
  }
  double* q = Q + e * THS;
#pragma unroll
  for (int s = 0; s < THS; ++s) q[s] = q[s] + dq[s];
}

// The same correction with one thread per (cell, mode) output: for large theta_S (3D, degree
// >= 4), where a thread holding a whole cell's time mean would spill, and for small meshes,
// which one thread per cell leaves on a few SMs.  Mode s has the digit a = s_d along dimension
// d and lies on the fibre base + b st of that dimension; every sum runs in the order of
// correct_linear_kernel, so the results are its bits.
template <int DIM, int NB>
__global__ void __launch_bounds__(128) correct_modes_kernel(double* Q, const double* Wb,
                                                            int wstride, int nx, int ny, int nz,
                                                            long long ncell, CorrParams cp) {
  constexpr int THS = ipow_c(NB, DIM);
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  grid_wait();
  if (i >= ncell * THS) return;
  const long long e = i / THS;
  const int s = (int)(i - e * THS);
  const Coords c = cell_coords(e, nx, ny);
  const double* w = Wb + e * wstride;
  double dq = 0.0;
#pragma unroll
  for (int dd = 0; dd < DIM; ++dd) {
    const int st = dd == 0 ? 1 : (dd == 1 ? NB : NB * NB);
    const int a = (s / st) % NB, base = s - a * st;
    double acc = 0.0;
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (b < a && ((a + b) & 1)) acc = fma(cp.D[a * kMaxNB + b], w[base + b * st], acc);
    dq = fma(cp.nu[dd], acc, dq);
    const Upwind uw = upwind_of(cp, dd);
    const double* wu = Wb + neighbour<DIM>(c, dd == 0 ? uw.up : 0, dd == 1 ? uw.up : 0,
                                           dd == 2 ? uw.up : 0, nx, ny, nz) * wstride;
    double to = 0.0, tu = 0.0;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      to = fma(uw.v[b], w[base + b * st], to);
      tu = fma(uw.v[b], wu[base + b * st], tu);
    }
    const double fo = uw.nf * to, fu = uw.nf * tu;
    const double fp = uw.up > 0 ? fu : fo, fm = uw.up > 0 ? fo : fu;
    dq = fma(-cp.ep[a], fp, dq);
    dq = fma(cp.em[a], fm, dq);
  }
  Q[e * THS + s] = Q[e * THS + s] + dq;
}

// Wb[e * thS + s] = W[e * thT + s], s < thS: the time means of a prediction, a thread per mode with
// four loads in flight (a warp per cell left most lanes idle at few modes: 96^3 Q1, 113 MB of W, 63
// -> 31 us)
__global__ void __launch_bounds__(256) time_means_kernel(const double* __restrict__ W, unsigned thT,
                                                         double* __restrict__ Wb, unsigned thS,
                                                         long long count) {
  const long long st = gridDim.x * 256LL;
  auto at = [&](long long i) {
    const long long e = i <= 0xFFFFFFFFLL ? (unsigned)i / thS : i / thS;
    return W[e * thT + (i - e * thS)];
  };
  long long i = blockIdx.x * 256LL + threadIdx.x;
  for (; i + 3 * st < count; i += 4 * st) {
    const double a = at(i), b = at(i + st), c = at(i + 2 * st), d = at(i + 3 * st);
    Wb[i] = a;
    Wb[i + st] = b;
    Wb[i + 2 * st] = c;
    Wb[i + 3 * st] = d;
  }
  for (; i < count; i += st) Wb[i] = at(i);
}

// FP64 operations of a 1D step per cell
double run1d_ops(int nb) { return nb * (2.0 * nb + 2.0) + nb * (0.25 * nb + 4.0); }
constexpr int kRun1dThreads = 768;

// 1D: k steps of a chunk of C cells per block and launch (temporal blocking).  With upwind face
// values a step reads two cells upstream (the time mean of the upstream neighbour reads one
// more), so a block that starts from 2k more cells upstream computes its own cells' k steps
// alone, each step on two cells fewer; blocks recompute each other's cells instead of
// exchanging them.  The sums are those of predict_fp64_kernel and correct_linear_kernel in the
// same order, so the states are theirs bit for bit.
//
// A step costs ~0.8 us of dependent FP64 operations and barriers whatever its cells, a launch
// ~1.7 us, and the FP64 pipe (2 FMA per clock and SM) adds the work of C + k cells on average;
// run1d_plan weighs the three.  Measured per step, against the whole run in one CTA (or, above
// 96 KB of state, one launch per kernel and step): 64 cells Q3 2.13 -> 1.14 us, 600 cells Q7 35.8
// -> 2.0, 1000 cells Q4 27.7 -> 1.6, 100000 cells Q3 37.4 -> 17.6.  Splitting the sums into two
// halves for a shorter chain gained nothing (1.21 us at 64 cells).
//
// A mesh of one block keeps its state in place (every read is ahead of the first barrier).
//
// One thread per (cell, mode); local cell u counts downstream, own cells are u >= 2k.
template <int NB>
__global__ void __launch_bounds__(kRun1dThreads) run1d_chunk_kernel(const double* Qin, double* Qout,
                                                           const double* __restrict__ P, int n,
                                                           int k, int C, CorrParams cp, int dir,
                                                           int nr) {
  extern __shared__ double sm1[];
  const int U = C + 2 * k;
  double* sQ = sm1;           // U x NB
  double* sW = sQ + U * NB;   // time means
  double* sF = sW + U * NB;   // value of the cell's downstream face
  const int tid = threadIdx.x, u = tid / NB, a = tid - u * NB;
  const bool act = u < U;
  // flow coordinate of the cell (periodic), its global cell
  int f = (int)((blockIdx.x * (long long)C + u - 2 * k) % n);
  f += f < 0 ? n : 0;
  const long long g = (long long)(dir > 0 ? f : n - 1 - f) * NB + a;
  double pr[2 * NB];  // this mode's row of the time-mean operator
#pragma unroll
  for (int i = 0; i < 2 * NB; ++i) pr[i] = i < nr * NB ? P[(size_t)a * nr * NB + i] : 0.0;
  const double nu = cp.nu[0], ep = cp.ep[a], em = cp.em[a];
  double tc[NB];  // the downstream face's trace
#pragma unroll
  for (int b = 0; b < NB; ++b) tc[b] = dir > 0 ? cp.ep[b] : cp.em[b];
  const double nf = cp.nu[0];
  double d[NB];  // row a of D, zero where a <= b or a + b is even
#pragma unroll
  for (int b = 0; b < NB; ++b) d[b] = a > b && ((a + b) & 1) ? cp.D[a * kMaxNB + b] : 0.0;
  grid_wait();
  double q = act ? Qin[g] : 0.0;
  if (act) sQ[tid] = q;
  __syncthreads();
  // the region's cells lo + 0, lo + 1: upstream and own for a > 0, own and upstream for a < 0
  const int r0 = nr == 2 ? (dir > 0 ? -NB : 0) : 0, r1 = dir > 0 ? 0 : -NB;
  for (int j = 1; j <= k; ++j) {
    if (act && u >= 2 * j - 1) {
      const double* x = sQ + u * NB;
      double acc = 0.0;
#pragma unroll
      for (int s2 = 0; s2 < NB; ++s2) acc = fma(pr[s2], x[r0 + s2], acc);
      if (nr == 2) {
#pragma unroll
        for (int s2 = 0; s2 < NB; ++s2) acc = fma(pr[NB + s2], x[r1 + s2], acc);
      }
      sW[tid] = acc;
    }
    __syncthreads();
    double v = 0.0;
    if (act && u >= 2 * j) {
      const double* w = sW + u * NB;
      double acc = 0.0;
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (d[b] != 0.0) acc = fma(d[b], w[b], acc);
      v = fma(nu, acc, 0.0);
    }
    if (tid < U && tid >= 2 * j - 1) {
      double t = 0.0;
#pragma unroll
      for (int b = 0; b < NB; ++b) t = fma(tc[b], sW[tid * NB + b], t);
      sF[tid] = nf * t;
    }
    __syncthreads();
    if (act && u >= 2 * j) {
      const double fp = sF[dir > 0 ? u : u - 1], fm = sF[dir > 0 ? u - 1 : u];
      v = fma(-ep, fp, v);
      v = fma(em, fm, v);
      q = q + v;
      sQ[tid] = q;
    }
    __syncthreads();
  }
  if (act && u >= 2 * k && blockIdx.x * (long long)C + u - 2 * k < n) Qout[g] = q;
}

int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return 1;
  return sms;
}

struct Run1dPlan {
  int C, launches;
};
// Cells per block and steps k per launch: the least of  max(chain, FP64 work) + launch / k  per
// step, in clocks (fitted to a sweep over C and k at 16 to 20000 cells, degrees 1 to 7; its
// choices are within 10% of the sweep's best).  Several blocks alternate between two states: an
// even number of launches, or a copy back; one block (C = n) keeps one state, which a few steps of
// a small mesh gain by (16 cells Q2, one step: 27.9 -> 25.6 us a call).
Run1dPlan run1d_plan(long long n, int nb, int nsteps, int sms) {
  const double chain = 1200.0 + 60.0 * nb, launch = 3000.0 + 100.0 * nb * nb;
  auto step = [&](long long C, int k) {
    const double blocks = std::ceil((double)n / C);
    const double work = std::ceil(blocks / std::max(1, sms)) * (C + k) * run1d_ops(nb) / 2.0;
    return std::max(chain, 700.0 + 1.5 * work);
  };
  int C = 1, k = 1;
  double cost = 1e300;
  for (int c : {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64})
    for (int q = 1; q <= 16 && q <= nsteps && (c + 2 * q) * nb <= kRun1dThreads; ++q) {
      const double t = step(c, q) + launch / q;
      if (t < cost) {
        cost = t;
        C = c;
        k = q;
      }
    }
  int launches = (nsteps + k - 1) / k;
  const bool copy = (launches & 1) && launches == nsteps;
  if ((launches & 1) && !copy) ++launches;
  if (nsteps <= 16 && (n + 2 * nsteps) * nb <= kRun1dThreads &&
      nsteps * step(n, nsteps) + launch < nsteps * step(C, k) + launches * launch + (copy ? 4000.0 : 0.0))
    return {(int)n, 1};
  return {C, launches};
}

template <int NB>
cudaError_t run1d_dispatch(const Grid& g, double* Q, double* Q2, const double* P, int nsteps,
                           const CorrParams& cp, cudaStream_t s) {
  const Run1dPlan pl = run1d_plan(g.ncell, NB, nsteps, device_sms());
  const int launches = pl.launches;
  const int dir = g.box.lo[0] < 0 ? 1 : (g.box.cnt[0] > 1 ? -1 : 1);
  const unsigned blocks = (unsigned)((g.ncell + pl.C - 1) / pl.C);
  double *in = Q, *out = pl.C < g.ncell ? Q2 : Q;
  for (int l = 0; l < launches; ++l) {
    const int k = nsteps / launches + (l < nsteps % launches);
    const int U = pl.C + 2 * k, threads = (U * NB + 31) / 32 * 32;
    const size_t smem = (size_t)U * (2 * NB + 1) * sizeof(double);
    const cudaError_t e = launch_dependent(true, run1d_chunk_kernel<NB>, blocks, threads, smem, s, in, out, P,
                                           (int)g.ncell, k, pl.C, cp, dir, g.box.cnt[0]);
    if (e != cudaSuccess) return e;
    std::swap(in, out);
  }
  cudaError_t e = cudaSuccess;
  if (in != Q)
    e = cudaMemcpyAsync(Q, in, (size_t)g.ncell * NB * sizeof(double), cudaMemcpyDeviceToDevice, s);
  return e;
}

// Rows of P per thread in 2D and 3D: up to 5 and a divisor of theta_S (4 of 3D Q4's 125 rows leave
// 3 of padding), so that meshes of a few thousand cells have warps for every SM; in 1D all NB.
// Measured against 16 rows (8 and 4 in 3D) by blocks of 128 threads, the time-mean prediction: 2D
// Q5 60^2 94.7 -> 43.5 us, Q3 256^2 138 -> 121, Q2 160^2 29 -> 21; 3D Q2 16^3 92 -> 53, Q3 8^3 164
// -> 97, Q3 48^3 5.88 -> 5.86 ms.
template <int DIM, int NB>
struct PredictRows {
  static constexpr int value = DIM == 1 ? NB
                               : NB == 1 ? 1
                               : NB == 2 ? 2
                               : NB == 3 ? 3
                               : NB == 5 ? 5
                                         : 4;
};

struct PredictGrid {
  int threads;
  size_t smem;
  dim3 grid;
  long long blocks, resident;  // resident: blocks that run at once on an SM
};
PredictGrid predict_grid(long long ncell, int K, int nout, int rows) {
  PredictGrid p;
  p.smem = (size_t)rows * K * sizeof(double);
  // one-warp blocks spread best; larger ones where each block's copy of its rows of P would
  // cost more than that gains (3D Q4, Q5: 32 to 55 KB)
  p.threads = p.smem <= 8 * 1024 ? 32 : p.smem <= 20 * 1024 ? 64 : 128;
  p.grid = dim3((unsigned)((ncell + p.threads - 1) / p.threads), (unsigned)((nout + rows - 1) / rows));
  p.blocks = (long long)p.grid.x * p.grid.y;
  p.resident = std::min({32LL, 2048LL / p.threads, 232448LL / (long long)(p.smem + 1024)});
  return p;
}

// The correction's form: a thread per mode below ~45 cells per SM, and where a cell's time means do
// not fit a thread.  The line lies between the sides at every degree (thread per mode against per
// cell, in us; 2D at 44 and 79 cells per SM, 3D at 38 and 70: 2D Q1 7.6 / 8.9 and 8.8 / 8.9, Q2 10.9 /
// 10.9 and 13.0 / 10.9, Q3 14.9 / 17.0 and 19.5 / 17.1, Q4 21.1 / 21.2 and 31.5 / 21.2, Q5 29.6 / 28.1
// and 48.0 / 29.3; 3D Q1 10.9 / 13.0 and 13.1 / 13.0, Q2 21.3 / 27.9 and 31.3 / 28.6, Q3 46.2 / 64.1 and
// 78.5 / 64.5).
bool correct_by_modes(int dim, int nb, long long ncell) {
  return (dim == 3 && nb >= 5) || ncell < 45LL * device_sms();
}
constexpr int kCorrectThreads = 128;
long long correct_blocks(bool modes, long long ncell, int ths) {
  return (ncell * (modes ? ths : 1) + kCorrectThreads - 1) / kCorrectThreads;
}

// Whether at most half of the correction's blocks that an SM can hold run on it.
template <int DIM, int NB>
bool correct_leaves_room(long long ncell) {
  auto resident = [](auto kern) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kCorrectThreads, 0) != cudaSuccess) n = 0;
    return n;
  };
  const bool modes = correct_by_modes(DIM, NB, ncell);
  long long room = 0;
  if (modes) {
    static const int n = resident(correct_modes_kernel<DIM, NB>);
    room = n;
  } else if constexpr (!(DIM == 3 && NB >= 5)) {
    static const int n = resident(correct_linear_kernel<DIM, NB>);
    room = n;
  }
  return 2 * correct_blocks(modes, ncell, ipow_c(NB, DIM)) <= room * device_sms();
}

template <int DIM, int NB, int CH>
cudaError_t predict_launch(const Grid& g, const double* Q, const double* P, int nout, double* W,
                           int wstride, cudaStream_t s) {
  const PredictGrid p = predict_grid(g.ncell, g.box.n * ipow_c(NB, DIM), nout, CH);
  auto kern = predict_fp64_kernel<DIM, NB, CH>;
  if (p.smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e != cudaSuccess) return e;
  }
  // Launched early, the blocks go to the SMs with room beside the correction of the step before.
  // Where that correction fills more than half of the chip, these are the few SMs that ran out
  // first, and a prediction that does not fill the chip by itself piles up there (3D Q3 16^3 424
  // against 262 us a step, Q5 10^3 875 against 691, 2D Q5 82^2 156 against 97, 1D Q11 100000 cells
  // 108 against 84; with room, 2D Q5 60^2, 3D Q2 14^3, it saves 6 to 8%).
  const int sms = device_sms();
  const bool early = correct_leaves_room<DIM, NB>(g.ncell) || 10 * p.blocks >= 9 * p.resident * sms;
  return launch_dependent(early, kern, p.grid, p.threads, p.smem, s, Q, P, nout, W, wstride, g.n[0],
                          g.n[1], g.n[2], g.ncell, g.box);
}

template <int DIM, int NB>
cudaError_t predict_dispatch_ch(const Grid& g, const double* Q, const double* P, int nout,
                                double* W, int wstride, cudaStream_t s) {
  if (g.box.n < 1 || g.box.n > ipow_c(2, DIM)) return cudaErrorInvalidValue;
  if constexpr (DIM == 3 && NB == 5) {
    // Few blocks of 40 KB: five rows per thread where the SM with the most blocks then has fewer
    // rows to sum and all blocks run at once, else four (a step, five against four rows: 9 x 10 x 8
    // 230 against 267 us, 11^3 347 against 405; 16^3 1151 against 943, 20^3 2374 against 1875).
    // Two warps of cells or fewer wait for their own sums: four (3 x 4 x 5 215 against 174).
    const int sms = device_sms();
    auto rows_on_sm = [&](const PredictGrid& p, int rows) {
      return (p.blocks + sms - 1) / sms * p.threads * rows;
    };
    const int K = g.box.n * ipow_c(NB, DIM);
    const PredictGrid p5 = predict_grid(g.ncell, K, nout, 5), p4 = predict_grid(g.ncell, K, nout, 4);
    if (g.ncell <= 64 || p5.blocks > p5.resident * sms || rows_on_sm(p5, 5) >= rows_on_sm(p4, 4))
      return predict_launch<DIM, NB, 4>(g, Q, P, nout, W, wstride, s);
  }
  return predict_launch<DIM, NB, PredictRows<DIM, NB>::value>(g, Q, P, nout, W, wstride, s);
}

template <int DIM, int NB>
cudaError_t correct_dispatch(const Grid& g, double* Q, const double* Wb, int wstride,
                             const CorrParams& cp, cudaStream_t s) {
  const int threads = kCorrectThreads;
  if (correct_by_modes(DIM, NB, g.ncell)) {
    const unsigned blocks = (unsigned)correct_blocks(true, g.ncell, ipow_c(NB, DIM));
    return launch_dependent(true, correct_modes_kernel<DIM, NB>, blocks, threads, 0, s, Q, Wb,
                            wstride, g.n[0], g.n[1], g.n[2], g.ncell, cp);
  } else if constexpr (!(DIM == 3 && NB >= 5)) {
    const unsigned blocks = (unsigned)correct_blocks(false, g.ncell, 1);
    return launch_dependent(true, correct_linear_kernel<DIM, NB>, blocks, threads, 0, s, Q, Wb,
                            wstride, g.n[0], g.n[1], g.n[2], g.ncell, cp);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

#define RIDG_DISPATCH_NB(DIM, FN, ...)                 \
  switch (nb) {                                        \
    case 1: return FN<DIM, 1>(__VA_ARGS__);            \
    case 2: return FN<DIM, 2>(__VA_ARGS__);            \
    case 3: return FN<DIM, 3>(__VA_ARGS__);            \
    case 4: return FN<DIM, 4>(__VA_ARGS__);            \
    default: break;                                    \
  }

cudaError_t launch_predict_fp64(const Grid& g, int nb, const double* Q, const double* P, int nout,
                                double* W, int wstride, cudaStream_t s) {
  if (g.dim == 1) {
    RIDG_DISPATCH_NB(1, predict_dispatch_ch, g, Q, P, nout, W, wstride, s)
    switch (nb) {
      case 5: return predict_dispatch_ch<1, 5>(g, Q, P, nout, W, wstride, s);
      case 6: return predict_dispatch_ch<1, 6>(g, Q, P, nout, W, wstride, s);
      case 7: return predict_dispatch_ch<1, 7>(g, Q, P, nout, W, wstride, s);
      case 8: return predict_dispatch_ch<1, 8>(g, Q, P, nout, W, wstride, s);
      case 9: return predict_dispatch_ch<1, 9>(g, Q, P, nout, W, wstride, s);
      case 10: return predict_dispatch_ch<1, 10>(g, Q, P, nout, W, wstride, s);
      case 11: return predict_dispatch_ch<1, 11>(g, Q, P, nout, W, wstride, s);
      case 12: return predict_dispatch_ch<1, 12>(g, Q, P, nout, W, wstride, s);
      default: break;
    }
  } else if (g.dim == 2) {
    RIDG_DISPATCH_NB(2, predict_dispatch_ch, g, Q, P, nout, W, wstride, s)
    switch (nb) {
      case 5: return predict_dispatch_ch<2, 5>(g, Q, P, nout, W, wstride, s);
      case 6: return predict_dispatch_ch<2, 6>(g, Q, P, nout, W, wstride, s);
      default: break;
    }
  } else if (g.dim == 3) {
    RIDG_DISPATCH_NB(3, predict_dispatch_ch, g, Q, P, nout, W, wstride, s)
    switch (nb) {
      case 5: return predict_dispatch_ch<3, 5>(g, Q, P, nout, W, wstride, s);
      case 6: return predict_dispatch_ch<3, 6>(g, Q, P, nout, W, wstride, s);
      default: break;
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_time_means(const double* W, int thT, double* Wb, int thS, long long ncell,
                              cudaStream_t s) {
  const long long count = ncell * thS;
  const unsigned blocks = (unsigned)std::min<long long>((count + 255) / 256, 8LL * device_sms());
  time_means_kernel<<<blocks, 256, 0, s>>>(W, (unsigned)thT, Wb, (unsigned)thS, count);
  return cudaGetLastError();
}

bool run1d_pays(const Grid& g, int nb, int nsteps) {
  if (nb == 1 && nsteps == 1) return g.ncell + 2 <= kRun1dThreads || g.ncell >= 100000;
  const double most = std::max(std::min(2000.0 * nb, 9000.0), 1250.0 * nb);
  return nb <= 2 || (double)g.ncell * run1d_ops(nb) / (2.0 * device_sms()) < most;
}

cudaError_t launch_run1d_fp64(const Grid& g, int nb, double* Q, double* Q2, const double* P,
                              int nsteps, const CorrParams& cp, cudaStream_t s) {
  if (g.dim != 1 || g.box.n < 1 || g.box.n > 2) return cudaErrorInvalidValue;
  switch (nb) {
    case 1: return run1d_dispatch<1>(g, Q, Q2, P, nsteps, cp, s);
    case 2: return run1d_dispatch<2>(g, Q, Q2, P, nsteps, cp, s);
    case 3: return run1d_dispatch<3>(g, Q, Q2, P, nsteps, cp, s);
    case 4: return run1d_dispatch<4>(g, Q, Q2, P, nsteps, cp, s);
    case 5: return run1d_dispatch<5>(g, Q, Q2, P, nsteps, cp, s);
    case 6: return run1d_dispatch<6>(g, Q, Q2, P, nsteps, cp, s);
    case 7: return run1d_dispatch<7>(g, Q, Q2, P, nsteps, cp, s);
    case 8: return run1d_dispatch<8>(g, Q, Q2, P, nsteps, cp, s);
    case 9: return run1d_dispatch<9>(g, Q, Q2, P, nsteps, cp, s);
    case 10: return run1d_dispatch<10>(g, Q, Q2, P, nsteps, cp, s);
    case 11: return run1d_dispatch<11>(g, Q, Q2, P, nsteps, cp, s);
    case 12: return run1d_dispatch<12>(g, Q, Q2, P, nsteps, cp, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_correct_linear(const Grid& g, int nb, double* Q, const double* Wbar,
                                  int wstride, const CorrParams& cp, cudaStream_t s) {
  if (g.dim == 1) {
    RIDG_DISPATCH_NB(1, correct_dispatch, g, Q, Wbar, wstride, cp, s)
    switch (nb) {
      case 5: return correct_dispatch<1, 5>(g, Q, Wbar, wstride, cp, s);
      case 6: return correct_dispatch<1, 6>(g, Q, Wbar, wstride, cp, s);
      case 7: return correct_dispatch<1, 7>(g, Q, Wbar, wstride, cp, s);
      case 8: return correct_dispatch<1, 8>(g, Q, Wbar, wstride, cp, s);
      case 9: return correct_dispatch<1, 9>(g, Q, Wbar, wstride, cp, s);
      case 10: return correct_dispatch<1, 10>(g, Q, Wbar, wstride, cp, s);
      case 11: return correct_dispatch<1, 11>(g, Q, Wbar, wstride, cp, s);
      case 12: return correct_dispatch<1, 12>(g, Q, Wbar, wstride, cp, s);
      default: break;
    }
  } else if (g.dim == 2) {
    RIDG_DISPATCH_NB(2, correct_dispatch, g, Q, Wbar, wstride, cp, s)
    switch (nb) {
      case 5: return correct_dispatch<2, 5>(g, Q, Wbar, wstride, cp, s);
      case 6: return correct_dispatch<2, 6>(g, Q, Wbar, wstride, cp, s);
      default: break;
    }
  } else if (g.dim == 3) {
    RIDG_DISPATCH_NB(3, correct_dispatch, g, Q, Wbar, wstride, cp, s)
    switch (nb) {
      case 5: return correct_dispatch<3, 5>(g, Q, Wbar, wstride, cp, s);
      case 6: return correct_dispatch<3, 6>(g, Q, Wbar, wstride, cp, s);
      default: break;
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace ridg
