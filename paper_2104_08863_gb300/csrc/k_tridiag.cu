// Wall-normal tridiagonal solves of Eq. 9: one system per (kx, kz) mode.
//
// Row j of mode (kx, kz), written as an M-matrix (all off-diagonals non-positive):
//     -a_j x_{j-1} + (a_j + c_j + sigma) x_j - c_j x_{j+1} = -F_j,
//     sigma = -(lambda_x(kx) + lambda_z(kz)) >= 0,
// with a_0 = c_{ny-1} = 0 (zero wall flux).
//
// PDD (Sec. 2.2, Eqs. 10-21): each system is cut into P blocks of m = ny/P rows; one thread
// owns one block, S systems share a CTA and neighbouring threads hold consecutive systems of one
// block index, so every row access is a coalesced segment of them.  Per block:
//   1. forward elimination of the block matrix A_i (Eq. 20) for the data and for the spike
//      a_1^i e_1;
//   2. the block's first-row values of x~, v, w (Eq. 20), summed up on the way;
//   3. the reduced interface system Z (Eqs. 18, 21) solved EXACTLY, framed entries included,
//      as a 2x2-block tridiagonal system over the P-1 interfaces by one thread per system;
//   4. a final backward sweep that folds the two neighbour values into the right-hand side,
//      which equals the correction x = x~ - Y y of Eq. 19.
// P = 1 is the Thomas algorithm (steps 1 and 4).
//
// The pivots use the cancellation-free "margin" recurrence: with beta_j the Thomas pivot and
// e_j = beta_j - c_j,  e_j = sigma + a_j e_{j-1} / beta_{j-1}  (all terms >= 0), so the
// weakly dominant low modes keep full relative accuracy.
//
// The singular (0, 0) mode and, in the FP32 forms, the lowest modes (FP64 systems) are skipped by
// the main pass and solved by extra CTAs at the head of its grid (low_modes.cuh).
#include "internal.h"
#include "low_modes.cuh"
#include "tridiag_scan.cuh"

namespace pp {

// ---- PDD with per-mode factors (FP64; FP32 blocks that do not fit in registers) ---------------
// The RHS-independent part of each block's elimination (pivots, spikes, first-row weights)
// depends only on the mode, so k_tridiag_setup computes it once per plan in FP64 and stores it
// in the solve's precision.  Per solve a thread then runs, for its m rows,
//   forward : g_j = -F_j + mult_j g_{j-1},  x~_{r0} += kappa_j g_j
//   exact reduced interface system (Eq. 21, framed entries included)
//   backward: x_j = (g_j + alpha gv_j + c_j x_{j+1}) rb_j
// FULL (FP64, FP64-issue bound) reads mult and kappa from tables; the lean FP32 variant
// (HBM bound) stores only rb and gv and recomputes mult_j = a_j rb_{j-1} and
// kappa_j = rb_j prod c_l rb_l with a few FP32 multiplies.  Rows are processed in chunks of
// CH so that a thread keeps CH independent loads in flight.

__device__ __forceinline__ void sys_to_mode(int sys, int ncols, int& kx, int& kz) {
  kz = sys / ncols;
  kx = sys - kz * ncols;
}

template <typename T, bool FULL>
__global__ void __launch_bounds__(256) k_tridiag_setup(Geometry g, int P, int m, const double* __restrict__ a,
                                                       const double* __restrict__ c,
                                                       const double* __restrict__ lamx,
                                                       const double* __restrict__ lamz, TriFactors<T> tf) {
  const int nsys = tf.nsys;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= (long long)nsys * P) return;
  const int b = (int)(tid / nsys), sys = (int)(tid - (long long)b * nsys);
  int kx, kz;
  sys_to_mode(sys, g.ncols, kx, kz);
  // (0,0) is solved elsewhere; give it a harmless positive shift so its factors stay finite
  const double sigma = (kx == 0 && kz == 0) ? 1.0 : -(lamx[kx] + lamz[kz]);
  const int r0 = b * m, r1 = r0 + m - 1;
  double e = a[r0] + sigma, gvv = a[r0], rbp = 0.0, run = 1.0, vF = 0.0, kap = 0.0;
  for (int i = 0; i < m; ++i) {
    const int j = r0 + i;
    double mult = 0.0;
    if (i > 0) {
      mult = a[j] * rbp;
      e = sigma + mult * e;
      gvv = mult * gvv;
    }
    const double rb = 1.0 / (c[j] + e);
    kap = run * rb;
    const size_t o = (size_t)j * nsys + sys;
    if constexpr (FULL) {
      tf.mult[o] = T(mult);
      tf.kappa[o] = T(kap);
    }
    tf.rb[o] = T(rb);
    tf.gv[o] = T(gvv);
    vF += kap * gvv;
    run *= c[j] * rb;
    rbp = rb;
  }
  const size_t ob = (size_t)b * nsys + sys;
  tf.vF[ob] = T(vF);
  tf.vL[ob] = T(gvv * rbp);
  tf.wF[ob] = T(kap * c[r1]);
  tf.wL[ob] = T(c[r1] * rbp);
}

template <typename T, bool FULL>
__global__ void __launch_bounds__(256) k_tridiag_factored(const __grid_constant__ Geometry g, int P, int m, int S, int low, int trunc,
                                                          const T* __restrict__ a, const T* __restrict__ c,
                                                          TriFactors<T> tf, cplx<T>* __restrict__ spec,
                                                          const __grid_constant__ SideArgs sd) {
  constexpr int CH = 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if ((int)blockIdx.x < sd.n) {
    low_system<T>(g, sd, spec, blockIdx.x);
    return;
  }
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int PS = P * S;
  T* xFr = sm;          T* xFi = sm + PS;      T* xLr = sm + 2 * PS;  T* xLi = sm + 3 * PS;
  T* alr = sm + 4 * PS; T* ali = sm + 5 * PS;  T* ber = sm + 6 * PS;  T* bei = sm + 7 * PS;
  T* y0r = sm + 8 * PS; T* y0i = sm + 9 * PS;  T* y1r = sm + 10 * PS; T* y1i = sm + 11 * PS;
  T* X01s = sm + 12 * PS; T* X11s = sm + 13 * PS;
  const int nsys = tf.nsys;
  const int tid = threadIdx.x;
  const int b = tid / S, s = tid - b * S;
  const int sys = ((int)blockIdx.x - sd.n) * S + s;
  int kx = 0, kz = 0;
  bool active = sys < nsys;
  if (active) {
    sys_to_mode(sys, g.ncols, kx, kz);
    if ((kx == 0 && kz == 0) || is_low(kx, kz, g.nz, low)) active = false;
  }
  const size_t rstride = (size_t)g.nz * g.pitch;
  cplx<T>* col = spec + (size_t)kz * g.pitch + kx;
  const int r0 = b * m;
  const int me = b * S + s;
  // ---- forward elimination and the block's end values of x~ ----
  cplx<T> xF = mk<T>(T(0), T(0)), xL = mk<T>(T(0), T(0));
  if (active) {
    cplx<T> gg = mk<T>(T(0), T(0));
    T rbp = T(0), run = T(1);
    for (int i0 = 0; i0 < m; i0 += CH) {
      cplx<T> F[CH];
      T t1[CH], t2[CH];
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        if (i0 + q < m) {
          const int j = r0 + i0 + q;
          const size_t o = (size_t)j * nsys + sys;
          F[q] = ld_c(col + (size_t)j * rstride);
          if constexpr (FULL) {
            t1[q] = tf.mult[o];
            t2[q] = tf.kappa[o];
          } else {
            t1[q] = tf.rb[o];
          }
        }
      }
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        if (i0 + q < m) {
          const int j = r0 + i0 + q;
          T mult, kap;
          if constexpr (FULL) {
            mult = t1[q];
            kap = t2[q];
          } else {
            const T rb = t1[q];
            mult = (i0 + q == 0) ? T(0) : a[j] * rbp;
            kap = run * rb;
            run *= c[j] * rb;
            rbp = rb;
          }
          gg = mk<T>(fma(mult, gg.x, -F[q].x), fma(mult, gg.y, -F[q].y));
          xF = mk<T>(fma(kap, gg.x, xF.x), fma(kap, gg.y, xF.y));
          F[q] = gg;
        }
      }
#pragma unroll
      for (int q = 0; q < CH; ++q)
        if (i0 + q < m) st_c(col + (size_t)(r0 + i0 + q) * rstride, F[q]);
    }
    T rbl;
    if constexpr (FULL) rbl = tf.rb[(size_t)(r0 + m - 1) * nsys + sys];
    else rbl = rbp;
    xL = mk<T>(gg.x * rbl, gg.y * rbl);
  }
  cplx<T> alpha = mk<T>(T(0), T(0)), beta = mk<T>(T(0), T(0));
  if (P > 1) {
    xFr[me] = xF.x; xFi[me] = xF.y; xLr[me] = xL.x; xLi[me] = xL.y;
    __syncthreads();
    if (b == 0 && active) {
      // exact reduced system over the interfaces, unknowns z_i = (L_i, F_{i+1})
      T pX01 = T(0);
      cplx<T> py0 = mk<T>(T(0), T(0));
      for (int i = 0; i < P - 1; ++i) {
        const int ii = i * S + s, in = (i + 1) * S + s;
        const size_t bi = (size_t)i * nsys + sys, bn = (size_t)(i + 1) * nsys + sys;
        // truncated (Sec. 2.2): the framed entries v_m^i and w_1^{i+1} of Z are dropped
        const T vLi = trunc ? T(0) : tf.vL[bi], wLi = tf.wL[bi], vFn = tf.vF[bn], wFi = tf.wF[bi];
        // eliminating z_{i-1} fills entry (0,1): L_i reaches F_{i+1} through L_{i-1} and F_i
        const T d01 = -wLi - vLi * wFi * pX01, d10 = -vFn;
        const T inv = T(1) / (T(1) - d01 * d10);
        const T X00 = inv, X01 = -d01 * inv, X10 = -d10 * inv, X11 = inv;
        const cplx<T> q0 = mk<T>(xLr[ii] + vLi * py0.x, xLi[ii] + vLi * py0.y);
        const cplx<T> q1 = mk<T>(xFr[in], xFi[in]);
        const cplx<T> y0 = mk<T>(X00 * q0.x + X01 * q1.x, X00 * q0.y + X01 * q1.y);
        const cplx<T> y1 = mk<T>(X10 * q0.x + X11 * q1.x, X10 * q0.y + X11 * q1.y);
        y0r[ii] = y0.x; y0i[ii] = y0.y; y1r[ii] = y1.x; y1i[ii] = y1.y;
        X01s[ii] = X01; X11s[ii] = X11;
        pX01 = X01;
        py0 = y0;
      }
      cplx<T> z1n = mk<T>(T(0), T(0));
      for (int i = P - 2; i >= 0; --i) {
        const int ii = i * S + s;
        const T tw = (i == P - 2 || trunc) ? T(0) : tf.wF[(size_t)(i + 1) * nsys + sys];
        const cplx<T> z0 = mk<T>(y0r[ii] + tw * z1n.x * X01s[ii], y0i[ii] + tw * z1n.y * X01s[ii]);
        const cplx<T> z1 = mk<T>(y1r[ii] + tw * z1n.x * X11s[ii], y1i[ii] + tw * z1n.y * X11s[ii]);
        alr[(i + 1) * S + s] = z0.x; ali[(i + 1) * S + s] = z0.y;   // alpha of block i+1 = L_i
        ber[ii] = z1.x; bei[ii] = z1.y;                              // beta of block i = F_{i+1}
        z1n = z1;
      }
    }
    __syncthreads();
    if (b > 0) alpha = mk<T>(alr[me], ali[me]);
    if (b < P - 1) beta = mk<T>(ber[me], bei[me]);
  }
  // ---- backward sweep with the neighbour values folded in ----
  if (active) {
    cplx<T> xn = beta;
    for (int i1 = m; i1 > 0; i1 -= CH) {
      cplx<T> G[CH];
      T rbv[CH], gvv[CH];
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        const int i = i1 - 1 - q;
        if (i >= 0) {
          const int j = r0 + i;
          const size_t o = (size_t)j * nsys + sys;
          G[q] = ld_c(col + (size_t)j * rstride);
          rbv[q] = tf.rb[o];
          gvv[q] = tf.gv[o];
        }
      }
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        const int i = i1 - 1 - q;
        if (i >= 0) {
          const T cj = c[r0 + i];
          const T tx = fma(cj, xn.x, fma(alpha.x, gvv[q], G[q].x));
          const T ty = fma(cj, xn.y, fma(alpha.y, gvv[q], G[q].y));
          xn = mk<T>(tx * rbv[q], ty * rbv[q]);
          G[q] = xn;
        }
      }
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        const int i = i1 - 1 - q;
        if (i >= 0) st_c(col + (size_t)(r0 + i) * rstride, G[q]);
      }
    }
  }
}

// ---- FP64 systems without partition on few modes ---------------------------------------------
// Thomas by scans: with the pivots in tables both sweeps are first-order linear recurrences with
// coefficients in (0, 1) (see low_modes.cuh), so 8 lanes take contiguous rows of one system each
// and the carries between them come from a 3-step scan of affine maps.  A warp holds 4 systems
// (64-byte row segments), a CTA 8, so that a few hundred systems reach every SM.  Per row the
// eliminated value and the running product of the coefficients (the weight of the carry) stay in the
// thread's own shared-memory column.
//
// Such a launch is bound by latency: one thread per system walks ny dependent rows twice (FP64
// FMA: 65 clocks) with 544 to 20,000 threads on the GPU.  It issues 13 FP64 instructions per row
// against 10 of the serial form, which stays for more modes.  32x32x32: 24.5 -> 12 us per launch
// with its event pair, 64x64x64: 43 -> 12 us; at 17,600 modes of 130 rows both take the same.
constexpr int kScan64Rows = 256;       // most rows (49 KB of shared memory)
constexpr int kScan64Systems = 20000;  // most modes

__global__ void __launch_bounds__(64) k_tridiag_scan64(const __grid_constant__ Geometry g, const double* __restrict__ c,
                                                        TriFactors<double> tf, cplx<double>* __restrict__ spec,
                                                        const __grid_constant__ SideArgs sd) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if ((int)blockIdx.x < sd.n) {
    low_system<double>(g, sd, spec, blockIdx.x);
    return;
  }
  const int lane = threadIdx.x & 31, l = lane >> 2;
  const int q = ((int)blockIdx.x - sd.n) * 8 + (threadIdx.x >> 5) * 4 + (lane & 3);   // over (kz, padded kx)
  const int kz = q / g.pitch, kx = q - kz * g.pitch;
  const bool active = kz < g.nz && kx < g.ncols && !(kx == 0 && kz == 0);
  const int ch = (g.ny + 7) / 8;
  const int lo = min(g.ny, l * ch), hi = active ? min(g.ny, lo + ch) : lo;
  double2* y = reinterpret_cast<double2*>(smem_raw) + threadIdx.x;                        // row lo + i at y[64 i]
  double* wt = reinterpret_cast<double*>(smem_raw) + (size_t)2 * 64 * ch + threadIdx.x;  // carry weights
  const size_t rstride = (size_t)g.nz * g.pitch, ns = (size_t)tf.nsys;
  cplx<double>* col = spec + (size_t)kz * g.pitch + kx;
  const double* mult = tf.mult + (size_t)kz * g.ncols + kx;
  const double* rb = tf.rb + (size_t)kz * g.ncols + kx;
  double A = 1.0;
  double2 B = make_double2(0.0, 0.0);
#pragma unroll 8
  for (int j = lo; j < hi; ++j) {
    const cplx<double> F = ld_c(col + (size_t)j * rstride);
    const double m = __ldg(mult + (size_t)j * ns);
    B = make_double2(fma(m, B.x, -F.x), fma(m, B.y, -F.y));
    A *= m;
    y[64 * (j - lo)] = B;
    wt[64 * (j - lo)] = A;
  }
  // the value entering this lane's rows, from the maps of the lanes before (UP) or after it
  auto carry = [&](bool up) {
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) {
      const double Ap = up ? __shfl_up_sync(0xffffffffu, A, 4 * d) : __shfl_down_sync(0xffffffffu, A, 4 * d);
      const double Bx = up ? __shfl_up_sync(0xffffffffu, B.x, 4 * d) : __shfl_down_sync(0xffffffffu, B.x, 4 * d);
      const double By = up ? __shfl_up_sync(0xffffffffu, B.y, 4 * d) : __shfl_down_sync(0xffffffffu, B.y, 4 * d);
      if (up ? l >= d : l + d < 8) {
        B = make_double2(fma(A, Bx, B.x), fma(A, By, B.y));
        A *= Ap;
      }
    }
    const double Bx = up ? __shfl_up_sync(0xffffffffu, B.x, 4) : __shfl_down_sync(0xffffffffu, B.x, 4);
    const double By = up ? __shfl_up_sync(0xffffffffu, B.y, 4) : __shfl_down_sync(0xffffffffu, B.y, 4);
    return (up ? l > 0 : l < 7) ? make_double2(Bx, By) : make_double2(0.0, 0.0);
  };
  const double2 gin = carry(true);
  A = 1.0;
  B = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int j = hi - 1; j >= lo; --j) {
    const double r = __ldg(rb + (size_t)j * ns), cr = c[j] * r, w = wt[64 * (j - lo)];
    const double2 v = y[64 * (j - lo)];
    B = make_double2(fma(cr, B.x, r * fma(w, gin.x, v.x)), fma(cr, B.y, r * fma(w, gin.y, v.y)));
    A *= cr;
    y[64 * (j - lo)] = B;
    wt[64 * (j - lo)] = A;
  }
  const double2 xin = carry(false);
#pragma unroll 4
  for (int j = lo; j < hi; ++j) {
    const double2 v = y[64 * (j - lo)];
    const double w = wt[64 * (j - lo)];
    st_c(col + (size_t)j * rstride, mk<double>(fma(w, xin.x, v.x), fma(w, xin.y, v.y)));
  }
}

// ---- FP32 PDD with thread-private blocks (P no power of two, or above 32) -------------------
// One thread owns one block of M rows of one system.  It copies its M rows into a private slice
// of shared memory with 8-byte cp.async (all M copies in flight, no register staging; layout
// [row][thread], so every shared access of a warp is conflict-free), eliminates forward while
// building the block's pivots and spike on the fly in FP32 (margin recurrence, reciprocal by
// MUFU plus one Newton step) and keeping them in registers, exchanges the block-end values
// through shared memory for the exact reduced interface system, and sweeps back, storing each
// result straight to global memory.  The spectrum crosses HBM once in each direction and no
// factor table is read.  Threads are numbered block-major (tid = b * S + s), so a warp's row
// accesses are S-system contiguous segments.

// Per-mode LU of the reduced interface system, built once per plan in FP64 (RHS-independent).
// For interface i (between blocks i and i+1) of system sys, entry k of
// table[(sys*(P-1) + i)*5 + k] (one contiguous record per system):
//   0: vL_i      the spike v of block i at its last row
//   1: inv_i     1 / (1 - d01 d10),  d01 = -wL_i - vL_i wF_i X01_{i-1},  d10 = -vF_{i+1}
//   2: X01_i     -d01 inv_i
//   3: X10_i     -d10 inv_i
//   4: wF_{i+1}  the spike w of block i+1 at its first row (0 for the last interface)
// One thread per system walks the blocks in order, keeping two blocks' spike values.
__device__ void block_spikes64(const double* a, const double* c, double sigma, int r0, int m, double& vF,
                               double& vL, double& wF, double& wL) {
  double e = a[r0] + sigma, gvv = a[r0], rbp = 0.0, run = 1.0, kap = 0.0;
  vF = 0.0;
  for (int i = 0; i < m; ++i) {
    const int j = r0 + i;
    if (i > 0) {
      const double mult = a[j] * rbp;
      e = sigma + mult * e;
      gvv = mult * gvv;
    }
    const double rb = 1.0 / (c[j] + e);
    kap = run * rb;
    vF += kap * gvv;
    run *= c[j] * rb;
    rbp = rb;
  }
  vL = gvv * rbp;
  wF = kap * c[r0 + m - 1];
  wL = c[r0 + m - 1] * rbp;
}

// Pivots of the modes solved apart, one thread per system of the list (low_system's order):
// rb[sys ny + j] = 1 / beta_j by the margin recurrence, in FP64.
struct LowSetup { int n, low; double* rb; };
__device__ void low_pivots(const Geometry& g, const LowSetup& ls, int sys, const double* __restrict__ a,
                           const double* __restrict__ c, const double* __restrict__ lamx,
                           const double* __restrict__ lamz) {
  if (sys < 1 || sys >= ls.n) return;
  const int kx = sys % (ls.low + 1), q = sys / (ls.low + 1);
  const int kz = q <= ls.low ? q : g.nz - (q - ls.low);
  const double sigma = -(lamx[kx] + lamz[kz]);
  double e = 0.0, r = 0.0;
  for (int j = 0; j < g.ny; ++j) {
    e = j > 0 ? sigma + a[j] * e * r : sigma;
    r = 1.0 / (c[j] + e);
    ls.rb[(size_t)sys * g.ny + j] = r;
  }
}
constexpr int kSetupThreads = 128;
static LowSetup low_setup(const DevTables& tb, int low) {
  return LowSetup{low < 1 ? 0 : (low + 1) * (2 * low + 1), low, tb.low_rb};   // low = 0: the (0, 0) mode only
}
static int low_blocks(const LowSetup& ls) { return (ls.n + kSetupThreads - 1) / kSetupThreads; }

__global__ void __launch_bounds__(kSetupThreads) k_low_setup(Geometry g, LowSetup ls, const double* __restrict__ a,
                                                            const double* __restrict__ c,
                                                            const double* __restrict__ lamx,
                                                            const double* __restrict__ lamz) {
  low_pivots(g, ls, blockIdx.x * blockDim.x + threadIdx.x, a, c, lamx, lamz);
}

// With the low modes' pivots by its first CTAs: both are chains of FP64 divisions, side by side.
__global__ void __launch_bounds__(kSetupThreads) k_reduced_setup(Geometry g, LowSetup ls, int nlow, int P, int m, int trunc,
                                                      const double* __restrict__ a,
                                                      const double* __restrict__ c, const double* __restrict__ lamx,
                                                      const double* __restrict__ lamz, float* __restrict__ tab) {
  if ((int)blockIdx.x < nlow) {
    low_pivots(g, ls, blockIdx.x * blockDim.x + threadIdx.x, a, c, lamx, lamz);
    return;
  }
  const int nsys = g.nz * g.ncols;
  const int sys = ((int)blockIdx.x - nlow) * blockDim.x + threadIdx.x;
  if (sys >= nsys) return;
  int kx, kz;
  sys_to_mode(sys, g.ncols, kx, kz);
  const double sigma = (kx == 0 && kz == 0) ? 1.0 : -(lamx[kx] + lamz[kz]);
  double vF0, vL0, wF0, wL0;
  block_spikes64(a, c, sigma, 0, m, vF0, vL0, wF0, wL0);
  double pX01 = 0.0;
  for (int i = 0; i < P - 1; ++i) {
    double vF1, vL1, wF1, wL1;
    block_spikes64(a, c, sigma, (i + 1) * m, m, vF1, vL1, wF1, wL1);
    // truncated (Sec. 2.2): without the framed entries v_m^i, w_1^{i+1} every interface is an
    // independent 2x2 system (no recurrence: vL and tw stored as 0)
    const double d01 = trunc ? -wL0 : -wL0 - vL0 * wF0 * pX01, d10 = -vF1;
    const double inv = 1.0 / (1.0 - d01 * d10);
    const double X01 = -d01 * inv, X10 = -d10 * inv;
    float* t = tab + ((size_t)sys * (P - 1) + i) * 5;
    t[0] = trunc ? 0.f : float(vL0);
    t[1] = float(inv);
    t[2] = float(X01);
    t[3] = float(X10);
    t[4] = (i + 1 < P - 1 && !trunc) ? float(wF1) : 0.f;
    pX01 = X01;
    vF0 = vF1; vL0 = vL1; wF0 = wF1; wL0 = wL1;
  }
}

// More CTAs to an SM at small heights, whose many interfaces make the reduced system a long chain
// (1536x536x486, 67 blocks of 8: solve 6155 us with 3 CTAs, 6077 with 4).
template <int M>
__global__ void __launch_bounds__(256, M <= 8 ? 4 : (M <= 12 ? 3 : 2))
    k_tridiag_reg(const __grid_constant__ Geometry g, int P, int S, int low, const float* __restrict__ a,
                  const float* __restrict__ c, const double* __restrict__ lamx, const double* __restrict__ lamz,
                  const float* __restrict__ rtab, cplx<float>* __restrict__ spec,
                  const __grid_constant__ SideArgs sd) {
  // shared: the interface arrays (6 x NT floats), the CTA's slice of the reduced-system table
  // (5 (P-1) S floats, [i][k][s]), then the blocks' rows [row][thread]
  extern __shared__ __align__(16) float red_s[];
  if ((int)blockIdx.x < sd.n) {
    low_system<float>(g, sd, spec, blockIdx.x);
    return;
  }
  enum { R_XFR, R_XFI, R_XLR, R_XLI, R_ZR, R_ZI };
  const int NT = P * S;
#define RED(k, idx) red_s[(k) * NT + (idx)]
  float* tsh = red_s + 6 * NT;
  float2* Xs = reinterpret_cast<float2*>(tsh + ((5 * (P - 1) * S + 1) & ~1));
  const int nsys = g.nz * g.ncols;
  const int tid = threadIdx.x;
  const int b = tid / S, s = tid - b * S;
  const int sys0 = ((int)blockIdx.x - sd.n) * S;
  const int sys = sys0 + s;
  int kx = 0, kz = 0;
  bool active = sys < nsys;
  if (active) {
    sys_to_mode(sys, g.ncols, kx, kz);
    if ((kx == 0 && kz == 0) || is_low(kx, kz, g.nz, low)) active = false;
  }
  const size_t rstride = (size_t)g.nz * g.pitch;
  float2* col = reinterpret_cast<float2*>(spec + (size_t)kz * g.pitch + kx);
  const int r0 = b * M;
  if (active) {
    const float2* src = col + (size_t)r0 * rstride;
#pragma unroll 1
    for (int i = 0; i < M; ++i, src += rstride) cp_async8(&Xs[i * NT + tid], src);
  }
  for (int q = tid; q < 5 * (P - 1) * S; q += NT) {   // the reduced-system table slice, [i][k][s]
    const int qs = q / (5 * (P - 1)), ik = q - qs * 5 * (P - 1);
    if (sys0 + qs < nsys) cp_async4(&tsh[ik * S + qs], &rtab[(size_t)(sys0 + qs) * 5 * (P - 1) + ik]);
  }
  float rbv[M], gvv[M];
  if (active) {
    const float sigma = float(-(lamx[kx] + lamz[kz]));
    cp_async_wait_all();
    float e = a[r0] + sigma, gv = a[r0], rb = rcp_nr(c[r0] + e);
    float run = 1.f;
    float2 gg = make_float2(0.f, 0.f);
    float2 xF = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < M; ++i) {
      const int j = r0 + i;
      const float cj = c[j];
      const float2 F = Xs[i * NT + tid];
      float mult = 0.f;
      if (i > 0) {
        mult = a[j] * rb;
        e = fmaf(mult, e, sigma);
        gv = mult * gv;
        rb = rcp_nr(cj + e);
      }
      gg = make_float2(fmaf(mult, gg.x, -F.x), fmaf(mult, gg.y, -F.y));
      Xs[i * NT + tid] = gg;
      rbv[i] = rb;
      gvv[i] = gv;
      const float kap = run * rb;
      xF.x = fmaf(kap, gg.x, xF.x);
      xF.y = fmaf(kap, gg.y, xF.y);
      run *= cj * rb;
    }
    RED(R_XFR, tid) = xF.x; RED(R_XFI, tid) = xF.y;
    RED(R_XLR, tid) = gg.x * rb; RED(R_XLI, tid) = gg.y * rb;
  } else {
    cp_async_wait_all();
  }
  float2 alpha = make_float2(0.f, 0.f), beta = make_float2(0.f, 0.f);
  if (P > 1) {
    __syncthreads();
    if (b == 0 && active) {
      // forward: y_i = [inv X01; X10 inv] (xL_i + vL_i y0_{i-1}, xF_{i+1}); y0 kept in R_Z, y1 in
      // the block's xF slot (no longer needed)
      float2 py0 = make_float2(0.f, 0.f);
      for (int i = 0; i < P - 1; ++i) {
        const int ii = i * S + s, in = ii + S;
        const float* t = tsh + i * 5 * S + s;
        const float vL = t[0], inv = t[S], X01 = t[2 * S], X10 = t[3 * S];
        const float q0x = fmaf(vL, py0.x, RED(R_XLR, ii)), q0y = fmaf(vL, py0.y, RED(R_XLI, ii));
        const float q1x = RED(R_XFR, in), q1y = RED(R_XFI, in);
        py0 = make_float2(fmaf(inv, q0x, X01 * q1x), fmaf(inv, q0y, X01 * q1y));
        RED(R_ZR, ii) = py0.x; RED(R_ZI, ii) = py0.y;
        RED(R_XFR, in) = fmaf(X10, q0x, inv * q1x); RED(R_XFI, in) = fmaf(X10, q0y, inv * q1y);
      }
      // backward: z1_i = y1_i + wF_{i+1} inv_i z1_{i+1}, z0_i = y0_i + wF_{i+1} X01_i z1_{i+1};
      // alpha of block i+1 = z0_i (stored in its R_XL slot), beta of block i = z1_i (R_Z slot)
      float2 z1n = make_float2(0.f, 0.f);
      for (int i = P - 2; i >= 0; --i) {
        const int ii = i * S + s, in = ii + S;
        const float* t = tsh + i * 5 * S + s;
        const float inv = t[S], X01 = t[2 * S], tw = t[4 * S];
        const float a0 = tw * X01, a1 = tw * inv;
        const float z0x = fmaf(a0, z1n.x, RED(R_ZR, ii)), z0y = fmaf(a0, z1n.y, RED(R_ZI, ii));
        z1n = make_float2(fmaf(a1, z1n.x, RED(R_XFR, in)), fmaf(a1, z1n.y, RED(R_XFI, in)));
        RED(R_XLR, in) = z0x; RED(R_XLI, in) = z0y;
        RED(R_ZR, ii) = z1n.x; RED(R_ZI, ii) = z1n.y;
      }
    }
    __syncthreads();
    if (b > 0) alpha = make_float2(RED(R_XLR, tid), RED(R_XLI, tid));
    if (b < P - 1) beta = make_float2(RED(R_ZR, tid), RED(R_ZI, tid));
  }
#undef RED
  if (active) {
    float2 xn = beta;
    float2* dst = col + (size_t)(r0 + M - 1) * rstride;
#pragma unroll
    for (int i = M - 1; i >= 0; --i) {
      const float cj = c[r0 + i];
      const float2 G = Xs[i * NT + tid];
      const float tx = fmaf(cj, xn.x, fmaf(alpha.x, gvv[i], G.x));
      const float ty = fmaf(cj, xn.y, fmaf(alpha.y, gvv[i], G.y));
      xn = make_float2(tx * rbv[i], ty * rbv[i]);
      *dst = xn;
      dst -= rstride;
    }
  }
}

// ---- FP32 PDD with the blocks in registers (P a power of two <= 32) --------------------------
// A CTA owns S = 256 / P consecutive systems of the flattened (kz, padded kx) index, thread
// (s, b) = (tid mod S, tid div S) block b of system s: it loads its M rows straight into registers
// (S-system row segments of 64 bytes or more, every load in flight before the first use), sweeps
// forward keeping per row rb_i gg_i, rb_i c_i and rb_i gv_i (4 registers), and after the reduced
// system sweeps back and stores each row as it is final.  Only the block-end values cross shared
// memory, twice: into system-major order, where the P interfaces of a system are P lanes of a
// warp and the reduced system is the pair of warp scans of tridiag_scan.cuh, and back.
//
// What bounds it is HBM and, on small grids, the latency of one load and two sweeps.  The form
// before staged the rows in shared memory and swept them there with 14 shared-memory wavefronts per
// warp and row (batch of 64 solves of 48 to 192 rows, a branch of the graph to each: 2678 us, 2520 with
// this kernel at every block height).
template <int M> constexpr int rows_min_ctas() { return M <= 8 ? 4 : (M <= 12 ? 3 : 2); }

template <int M>
__global__ void __launch_bounds__(256, rows_min_ctas<M>())
    k_tridiag_rows(const __grid_constant__ Geometry g, int lgP, int low, const float* __restrict__ a, const float* __restrict__ c,
                   const double* __restrict__ lamx, const double* __restrict__ lamz, const float* __restrict__ rtab,
                   cplx<float>* __restrict__ spec, int kx_lo, int kx_hi, int width, const __grid_constant__ SideArgs sd) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if ((int)blockIdx.x < sd.n) {
    low_system<float>(g, sd, spec, blockIdx.x);
    return;
  }
  constexpr int MS = M | 1;   // odd stride of a block's (a, c) pairs
  const int P = 1 << lgP, S = 256 >> lgP;
  const int tid = threadIdx.x;
  const int s = tid & (S - 1), b = tid >> (8 - lgP);
  float4* ex = reinterpret_cast<float4*>(smem_raw);                   // [s][b], stride P + 1
  float* rec = reinterpret_cast<float*>(ex + (size_t)S * (P + 1));    // interface records [k][tid]
  float2* ac = reinterpret_cast<float2*>(rec + 5 * 256);              // [b][i]
  const int idx0 = ((int)blockIdx.x - sd.n) * S, total = g.nz * width;
  // mode of system index q of the flattened (kz, kx - kx_lo) order; false for padding, columns
  // outside the launch and the modes solved apart
  auto mode = [&](int q, int& kx, int& kz) {
    kz = q / width;
    kx = kx_lo + q - kz * width;
    return q < total && kx < kx_hi && !(kx == 0 && kz == 0) && !is_low(kx, kz, g.nz, low);
  };
  int kx, kz;
  const bool active = mode(idx0 + s, kx, kz);
  const size_t rstride = (size_t)g.nz * g.pitch;
  float2* p = reinterpret_cast<float2*>(spec) + (size_t)kz * g.pitch + kx + (size_t)b * M * rstride;
  float2 v[M];
  if (active) {
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = __ldcg(p + (size_t)i * rstride);
  }
  // interface role: thread (s2, b2) of the system-major order, its record fetched meanwhile
  const int s2 = tid >> lgP, b2 = tid & (P - 1);
  bool iface = false;
  if (P > 1 && b2 < P - 1) {
    int kx2, kz2;
    iface = mode(idx0 + s2, kx2, kz2);
    if (iface) {
      const float* t = rtab + ((size_t)(kz2 * g.ncols + kx2) * (P - 1) + b2) * 5;
#pragma unroll
      for (int k = 0; k < 5; ++k) cp_async4(rec + k * 256 + tid, t + k);
    }
  }
  for (int j = tid; j < g.ny; j += 256) {
    const int bj = j / M;
    ac[bj * MS + j - bj * M] = make_float2(a[j], c[j]);
  }
  const float sigma = active ? float(-(lamx[kx] + lamz[kz])) : 0.f;
  __syncthreads();
  const float2* co = ac + b * MS;
  float rcv[M], rgv[M];
  float2 xF = make_float2(0.f, 0.f), xL = make_float2(0.f, 0.f);
  if (active) {
    float2 cf = co[0];
    float e = cf.x + sigma, gv = cf.x, rb = rcp_nr(cf.y + e);
    float run = 1.f;
    float2 gg = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < M; ++i) {
      float mult = 0.f;
      if (i > 0) {
        cf = co[i];
        mult = cf.x * rb;
        e = fmaf(mult, e, sigma);
        gv = mult * gv;
        rb = rcp_nr(cf.y + e);
      }
      gg = make_float2(fmaf(mult, gg.x, -v[i].x), fmaf(mult, gg.y, -v[i].y));
      v[i] = make_float2(gg.x * rb, gg.y * rb);
      const float crb = cf.y * rb;
      rcv[i] = crb;
      rgv[i] = gv * rb;
      const float kap = run * rb;
      xF.x = fmaf(kap, gg.x, xF.x);
      xF.y = fmaf(kap, gg.y, xF.y);
      run *= crb;
    }
    xL = v[M - 1];
  }
  float2 alpha = make_float2(0.f, 0.f), beta = make_float2(0.f, 0.f);
  if (P > 1) {
    ex[s * (P + 1) + b] = make_float4(xF.x, xF.y, xL.x, xL.y);
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    float4* mine = ex + s2 * (P + 1) + b2;
    const float4 x = *mine;
    float vL = 0.f, inv = 0.f, X01 = 0.f, X10 = 0.f, tw = 0.f;
    if (iface) {
      vL = rec[tid]; inv = rec[256 + tid]; X01 = rec[512 + tid]; X10 = rec[768 + tid]; tw = rec[1024 + tid];
    }
    float2 al, be;
    scan_interfaces(P, b2, make_float2(x.x, x.y), make_float2(x.z, x.w), vL, inv, X01, X10, tw, al, be);
    *mine = make_float4(al.x, al.y, be.x, be.y);
    __syncthreads();
    const float4 y = ex[s * (P + 1) + b];
    alpha = make_float2(y.x, y.y);
    beta = make_float2(y.z, y.w);
  }
  if (active) {
    float2 xn = beta;
#pragma unroll
    for (int i = M - 1; i >= 0; --i) {
      xn = make_float2(fmaf(rcv[i], xn.x, fmaf(rgv[i], alpha.x, v[i].x)),
                       fmaf(rcv[i], xn.y, fmaf(rgv[i], alpha.y, v[i].y)));
      p[(size_t)i * rstride] = xn;
    }
  }
}

// ---- FP32 PDD on tiles in shared memory (P >= 16, blocks of 12 rows and more) -------------------
// The rows kernel's blocks and order, with the S = NT / P systems of a CTA staged in shared memory
// as [row][s] by 16-byte asynchronous copies.  A thread keeps only 1/beta_i per row in registers
// (64 in all), so that 1024 threads are resident where 4 registers per row allow 512: 32 warps hide
// the sweeps' latencies and one CTA's copies overlap the other's sweeps.  The forward sweep stores rb_i gg_i in place; once alpha
// is known a second one adds alpha rb_i gv_i (gv_i = a_i rb_{i-1} gv_{i-1} again), and the backward
// sweep writes x_i to global memory as it goes: the operations of the rows kernel, bit for bit.
//
// What bounds it is the rate at which HBM serves row segments that lie nz pitch * 8 bytes apart
// (6.4 MB at 1536x768x1024): an in-place copy in this order runs at 4.1 TB/s with 64-byte segments
// and at 6.7 TB/s with 128-byte ones, so a CTA takes at least 16 systems: 512 threads at P = 32
// (M = 24: 113,152 bytes of shared memory, 98,304 of them rows; two CTAs fill 224 of an SM's 228 KB), else 256.  Per pass, against the rows kernel (4
// registers per row, 8 systems per CTA at P = 32): 1536x768x1024 2.13 against 2.58 ms,
// 768x384x512 246 against 250 us; with 512 threads at P = 16 267 us.  Copies of 8 bytes cost half
// as much again (3.0 ms), stores through shared memory 0.27 ms.  At P <= 8 the rows kernel's segments
// are 256 bytes and more: 384x192x256 alone takes 35 against 38 us here, but a batch of 64 solves
// side by side 2736 us with this kernel and 2520 with that one (its CTAs need little shared memory).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}

template <int M, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT)
    k_tridiag_tile(const __grid_constant__ Geometry g, int lgP, int low, const float* __restrict__ a, const float* __restrict__ c,
                   const double* __restrict__ lamx, const double* __restrict__ lamz, const float* __restrict__ rtab,
                   cplx<float>* __restrict__ spec, int kx_lo, int kx_hi, int width, const __grid_constant__ SideArgs sd) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if ((int)blockIdx.x < sd.n) {
    low_system<float>(g, sd, spec, blockIdx.x);
    return;
  }
  static_assert(M % 2 == 0, "whole rounds of pair copies");
  constexpr int MS = M | 1, LGNT = NT == 512 ? 9 : 8;   // odd stride of a block's (a, c) pairs
  const int P = 1 << lgP, lgS = LGNT - lgP, S = 1 << lgS;
  const int tid = threadIdx.x;
  const int s = tid & (S - 1), b = tid >> lgS;
  float2* tile = reinterpret_cast<float2*>(smem_raw);                 // [row][s]
  float4* ex = reinterpret_cast<float4*>(tile + (size_t)M * NT);      // [s][b], stride P + 1
  float2* ac = reinterpret_cast<float2*>(ex + (size_t)S * (P + 1));   // [b][i]
  const int idx0 = ((int)blockIdx.x - sd.n) * S, total = g.nz * width;
  // mode of index q of the flattened (kz, kx - kx_lo) order; false for padding, columns outside the
  // launch and the modes solved apart
  auto mode = [&](int q, int& kx, int& kz) {
    kz = q / width;
    kx = kx_lo + q - kz * width;
    return q < total && kx < kx_hi && !(kx == 0 && kz == 0) && !is_low(kx, kz, g.nz, low);
  };
  const size_t rstride = (size_t)g.nz * g.pitch;
  {   // a pair of systems per copy; width is even, so a pair never crosses a row of the spectrum
    const int q = idx0 + 2 * (tid & (S / 2 - 1)), r0 = tid >> (lgS - 1);
    if (q < total) {
      const int kz = q / width;
      const float2* src = reinterpret_cast<const float2*>(spec) + (size_t)kz * g.pitch + kx_lo + (q - kz * width) +
                          (size_t)r0 * rstride;
      float2* dst = tile + 2 * tid;
      const size_t step = (size_t)(2 * P) * rstride;   // 2 P rows per round of the CTA
#pragma unroll
      for (int n = 0; n < M / 2; ++n) cp_async16(dst + (size_t)n * 2 * NT, src + n * step);
    }
  }
  int kx, kz;
  const bool active = mode(idx0 + s, kx, kz);
  for (int j = tid; j < g.ny; j += NT) {
    const int bj = j / M;
    ac[bj * MS + j - bj * M] = make_float2(a[j], c[j]);
  }
  const float sigma = active ? float(-(lamx[kx] + lamz[kz])) : 0.f;
  cp_async_wait_all();
  __syncthreads();
  const float2* co = ac + b * MS;
  float2* rows = tile + (size_t)b * M * S + s;
  float rbv[M];
  float2 xF = make_float2(0.f, 0.f), xL = make_float2(0.f, 0.f);
  if (active) {
    float2 cf = co[0];
    float e = cf.x + sigma, rb = rcp_nr(cf.y + e), run = 1.f;
    float2 gg = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < M; ++i) {
      const float2 F = rows[i * S];
      float mult = 0.f;
      if (i > 0) {
        cf = co[i];
        mult = cf.x * rb;
        e = fmaf(mult, e, sigma);
        rb = rcp_nr(cf.y + e);
      }
      gg = make_float2(fmaf(mult, gg.x, -F.x), fmaf(mult, gg.y, -F.y));
      xL = make_float2(gg.x * rb, gg.y * rb);
      rows[i * S] = xL;
      rbv[i] = rb;
      const float kap = run * rb;
      xF.x = fmaf(kap, gg.x, xF.x);
      xF.y = fmaf(kap, gg.y, xF.y);
      run *= cf.y * rb;
    }
  }
  ex[s * (P + 1) + b] = make_float4(xF.x, xF.y, xL.x, xL.y);
  const int s2 = tid >> lgP, b2 = tid & (P - 1);   // interface role, system-major
  float vL = 0.f, inv = 0.f, X01 = 0.f, X10 = 0.f, tw = 0.f;
  int kx2, kz2;
  if (b2 < P - 1 && mode(idx0 + s2, kx2, kz2)) {
    const float* r = rtab + ((size_t)(kz2 * g.ncols + kx2) * (P - 1) + b2) * 5;
    vL = __ldg(r); inv = __ldg(r + 1); X01 = __ldg(r + 2); X10 = __ldg(r + 3); tw = __ldg(r + 4);
  }
  __syncthreads();
  float4* mine = ex + s2 * (P + 1) + b2;
  const float4 x = *mine;
  float2 al, be;
  scan_interfaces(P, b2, make_float2(x.x, x.y), make_float2(x.z, x.w), vL, inv, X01, X10, tw, al, be);
  *mine = make_float4(al.x, al.y, be.x, be.y);
  __syncthreads();
  if (active) {
    const float4 y = ex[s * (P + 1) + b];
    float gv = co[0].x;
#pragma unroll
    for (int i = 0; i < M; ++i) {
      if (i > 0) gv = co[i].x * rbv[i - 1] * gv;
      const float rgv = gv * rbv[i];
      const float2 q = rows[i * S];
      rows[i * S] = make_float2(fmaf(rgv, y.x, q.x), fmaf(rgv, y.y, q.y));
    }
    float2 xn = make_float2(y.z, y.w);
    float2* p = reinterpret_cast<float2*>(spec) + (size_t)kz * g.pitch + kx + (size_t)(b * M + M - 1) * rstride;
#pragma unroll
    for (int i = M - 1; i >= 0; --i, p -= rstride) {
      const float2 q = rows[i * S];
      const float crb = co[i].y * rbv[i];
      xn = make_float2(fmaf(crb, xn.x, q.x), fmaf(crb, xn.y, q.y));
      *p = xn;
    }
  }
}

// ------------------------------------------------------------------------------ launchers
template <typename K>
static cudaError_t prep(K kernel, size_t smem) {
  return ensure_smem_limit((const void*)kernel, smem);
}

// The modes solved apart (low_modes.cuh): as extra CTAs of the main launch, or (side_apart, ny > 3072) as a
// launch of their own before it.
template <typename TD>
__global__ void __launch_bounds__(128) k_tridiag_side(const __grid_constant__ Geometry g,
                                                      const __grid_constant__ SideArgs sd,
                                                      cplx<TD>* __restrict__ spec) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  low_system<TD>(g, sd, spec, blockIdx.x);
}

// Groups of sd for CTAs of `threads` threads: a warp per system up to 256 rows, else 128 threads; at
// most two systems to a CTA, since the groups of a CTA share the two FP64 instructions per clock of
// their SM (162x90x108 solve 39.2 -> 37.2 us, 192x96x192 pass 18 -> 16 us with eight; the batch of 64 solves
// does not see the difference).
static void side_groups(const Geometry& g, SideArgs& sd, int threads) {
  const int whole = threads & ~31;
  sd.threads = g.ny <= 256 ? 32 : (whole < 128 ? whole : 128);
  sd.per = whole / sd.threads;
  if (sd.per > kLowMaxGroups) sd.per = kLowMaxGroups;
  while (sd.per > 1 && (size_t)16 * g.ny * sd.per > kSideFusedBytes) --sd.per;
  sd.n = (sd.nsys + sd.per - 1) / sd.per;
}

// sd for a main launch of CTAs of `threads` threads (n = 0 after a launch of its own); smem
// raised to the work area.
template <typename TD>
static cudaError_t prepare_side(const Geometry& g, SideArgs& sd, int threads, size_t& smem, cplx<TD>* spec,
                                cudaStream_t st) {
  sd.n = 0;
  if (sd.nsys == 0) return cudaSuccess;
  if (!side_apart(g)) {
    side_groups(g, sd, threads);
    const size_t need = (size_t)16 * g.ny * sd.per;
    if (smem < need) smem = need;
    return cudaSuccess;
  }
  side_groups(g, sd, 128);
  const size_t need = (size_t)16 * g.ny;
  cudaError_t e = prep(k_tridiag_side<TD>, need);
  if (e != cudaSuccess) return e;
  k_tridiag_side<TD><<<sd.n, 128, need, st>>>(g, sd, spec);
  sd.n = 0;
  return cudaGetLastError();
}

SideArgs side_args(const DevTables& tb, int low, GaugeMode gauge) {
  SideArgs sd;
  sd.nsys = low >= 0 ? (low + 1) * (2 * low + 1) : 1;
  sd.n = sd.per = sd.threads = 0;   // set for each launch (prepare_side)
  sd.low = low;
  sd.gauge = (int)gauge;
  sd.a = tb.d.a;
  sd.c = tb.d.c;
  sd.rb = tb.low_rb;
  sd.dy = tb.dy;
  sd.h = tb.h;
  sd.acc = tb.acc;
  return sd;
}

cudaError_t launch_low_setup(const Geometry& g, const DevTables& tb, int low, cudaStream_t st) {
  const LowSetup ls = low_setup(tb, low);
  if (ls.n == 0) return cudaSuccess;
  k_low_setup<<<low_blocks(ls), kSetupThreads, 0, st>>>(g, ls, tb.d.a, tb.d.c, tb.lamx, tb.lamz);
  return cudaGetLastError();
}

cudaError_t launch_tridiag_setup(const Geometry& g, const DevTables& tb, int parts, cudaStream_t st) {
  if (tb.tri_d.nsys) {
    const long long n = (long long)tb.tri_d.nsys * parts;
    k_tridiag_setup<double, true><<<(int)((n + 255) / 256), 256, 0, st>>>(g, parts, g.ny / parts, tb.d.a, tb.d.c,
                                                                          tb.lamx, tb.lamz, tb.tri_d);
  }
  if (tb.tri_f.nsys) {
    const long long n = (long long)tb.tri_f.nsys * parts;
    k_tridiag_setup<float, false><<<(int)((n + 255) / 256), 256, 0, st>>>(g, parts, g.ny / parts, tb.d.a, tb.d.c,
                                                                          tb.lamx, tb.lamz, tb.tri_f);
  }
  return cudaGetLastError();
}

template <typename T, bool FULL>
static cudaError_t launch_factored(const Geometry& g, const T* a, const T* c, const TriFactors<T>& tf, int parts,
                                   int low, bool trunc, cplx<T>* spec, SideArgs sd, cudaStream_t st) {
  int S = 256 / parts;
  if (S < 1) S = 1;
  if (S > 32) S = 32;
  size_t smem = (size_t)14 * parts * S * sizeof(T);
  const int blocks = (tf.nsys + S - 1) / S;
  auto kern = k_tridiag_factored<T, FULL>;
  cudaError_t e;
  if ((e = prepare_side<T>(g, sd, parts * S, smem, spec, st)) != cudaSuccess) return e;
  if ((e = prep(kern, smem)) != cudaSuccess) return e;
  kern<<<sd.n + blocks, parts * S, smem, st>>>(g, parts, g.ny / parts, S, low, trunc ? 1 : 0, a, c, tf, spec, sd);
  return cudaGetLastError();
}

size_t reduced_table_bytes(const Geometry& g, int parts) {
  return parts > 1 ? (size_t)5 * (parts - 1) * g.nz * g.ncols * sizeof(float) : 0;
}

cudaError_t launch_reduced_setup(const Geometry& g, const DevTables& tb, int parts, bool trunc, int low, float* tab,
                                 cudaStream_t st) {
  if (parts <= 1) return launch_low_setup(g, tb, low, st);
  const int nsys = g.nz * g.ncols;
  const LowSetup ls = low_setup(tb, low);
  const int nlow = low_blocks(ls);
  k_reduced_setup<<<nlow + (nsys + kSetupThreads - 1) / kSetupThreads, kSetupThreads, 0, st>>>(
      g, ls, nlow, parts, g.ny / parts, trunc ? 1 : 0, tb.d.a, tb.d.c, tb.lamx, tb.lamz, tab);
  return cudaGetLastError();
}

// The launch's columns: a whole row with its padding, so that the systems of a CTA start on a
// 64-byte boundary (S >= 8).
static int launch_width(const Geometry& g, int kx_lo, int kx_hi) { return (kx_hi == g.ncols ? g.pitch : kx_hi) - kx_lo; }
static int log2_of(int P) {
  int l = 0;
  while ((1 << l) < P) ++l;
  return l;
}

template <int M>
static cudaError_t launch_rows(const Geometry& g, const DevTables& tb, int parts, int low, cplx<float>* spec,
                               SideArgs sd, cudaStream_t st, int kx_lo, int kx_hi) {
  const int S = 256 / parts, width = launch_width(g, kx_lo, kx_hi), blocks = (g.nz * width + S - 1) / S;
  size_t smem = (size_t)S * (parts + 1) * 16 + 5 * 256 * 4 + (size_t)parts * (M | 1) * 8;
  cudaError_t e = prepare_side<float>(g, sd, 256, smem, spec, st);
  if (e != cudaSuccess) return e;
  if ((e = prep(k_tridiag_rows<M>, smem)) != cudaSuccess) return e;
  k_tridiag_rows<M><<<sd.n + blocks, 256, smem, st>>>(g, log2_of(parts), low, tb.f.a, tb.f.c, tb.lamx, tb.lamz,
                                                      tb.red_f, spec, kx_lo, kx_hi, width, sd);
  return cudaGetLastError();
}

template <int M, int NT>
static cudaError_t launch_tile(const Geometry& g, const DevTables& tb, int parts, int low, cplx<float>* spec,
                               SideArgs sd, cudaStream_t st, int kx_lo, int kx_hi) {
  const int S = NT / parts, width = launch_width(g, kx_lo, kx_hi), blocks = (g.nz * width + S - 1) / S;
  size_t smem = (size_t)M * NT * 8 + (size_t)S * (parts + 1) * 16 + (size_t)parts * (M | 1) * 8;
  cudaError_t e = prepare_side<float>(g, sd, 256, smem, spec, st);
  if (e != cudaSuccess) return e;
  auto kern = k_tridiag_tile<M, NT>;
  if ((e = prep(kern, smem)) != cudaSuccess) return e;
  kern<<<sd.n + blocks, NT, smem, st>>>(g, log2_of(parts), low, tb.f.a, tb.f.c, tb.lamx, tb.lamz, tb.red_f, spec, kx_lo,
                                        kx_hi, width, sd);
  return cudaGetLastError();
}

cudaError_t launch_tridiag_reg_f32(const Geometry& g, const DevTables& tb, int parts, int low_modes,
                                   cplx<float>* spec, SideArgs sd, cudaStream_t st, int kx_lo, int kx_hi) {
  if (!reg_kernel_ok(g.ny, parts)) return cudaErrorNotSupported;
  const int m = g.ny / parts;
  const int S = reg_systems_per_cta(parts);
  if (kx_hi < 0) kx_hi = g.ncols;
  const bool whole = kx_lo == 0 && kx_hi == g.ncols;
  if (kx_lo < 0 || kx_hi > g.ncols || kx_hi <= kx_lo) return cudaErrorInvalidValue;
  if (!whole && (!scan_tridiag_ok(g.ny, parts) || kx_lo % S)) return cudaErrorNotSupported;
  if (scan_tridiag_ok(g.ny, parts)) {   // P a power of two <= 32
    // P >= 16 with blocks of at least 12 rows: tiles in shared memory; else in registers (both
    // sides measured, see the two kernels)
    if (parts >= 16) {
      switch (m) {
#define PP_TILE_CASE(MM)                                                                           \
  case MM:                                                                                         \
    return parts == 32 ? launch_tile<MM, 512>(g, tb, parts, low_modes, spec, sd, st, kx_lo, kx_hi) \
                       : launch_tile<MM, 256>(g, tb, parts, low_modes, spec, sd, st, kx_lo, kx_hi);
        PP_TILE_CASE(12) PP_TILE_CASE(16) PP_TILE_CASE(24)
        default: break;
      }
    }
#define PP_ROWS_CASE(MM) \
  case MM: return launch_rows<MM>(g, tb, parts, low_modes, spec, sd, st, kx_lo, kx_hi);
    switch (m) {
      PP_ROWS_CASE(1) PP_ROWS_CASE(2) PP_ROWS_CASE(3) PP_ROWS_CASE(4) PP_ROWS_CASE(6) PP_ROWS_CASE(8)
      PP_ROWS_CASE(12) PP_ROWS_CASE(16) PP_ROWS_CASE(24)
      default: break;
    }
#undef PP_TILE_CASE
#undef PP_ROWS_CASE
  }
  const int nt = parts * S;
  const size_t tabf = ((size_t)5 * (parts - 1) * S + 1) & ~(size_t)1;
  size_t smem = (size_t)6 * nt * sizeof(float) + tabf * sizeof(float) + (size_t)m * 8 * nt;
  const int nsys = g.nz * g.ncols;
  const int blocks = (nsys + S - 1) / S;
  const cudaError_t es = prepare_side<float>(g, sd, nt, smem, spec, st);
  if (es != cudaSuccess) return es;
#define PP_REG_CASE(MM)                                                                                         \
  case MM: {                                                                                                    \
    cudaError_t e = prep(k_tridiag_reg<MM>, smem);                                                              \
    if (e != cudaSuccess) return e;                                                                             \
    k_tridiag_reg<MM><<<sd.n + blocks, nt, smem, st>>>(g, parts, S, low_modes, tb.f.a, tb.f.c, tb.lamx,         \
                                                       tb.lamz, tb.red_f, spec, sd);                            \
    break;                                                                                                      \
  }
  switch (m) {
    PP_REG_CASE(1) PP_REG_CASE(2) PP_REG_CASE(3) PP_REG_CASE(4) PP_REG_CASE(5) PP_REG_CASE(6)
    PP_REG_CASE(7) PP_REG_CASE(8) PP_REG_CASE(9) PP_REG_CASE(10) PP_REG_CASE(11) PP_REG_CASE(12)
    PP_REG_CASE(13) PP_REG_CASE(14) PP_REG_CASE(15) PP_REG_CASE(16) PP_REG_CASE(17) PP_REG_CASE(18)
    PP_REG_CASE(19) PP_REG_CASE(20) PP_REG_CASE(21) PP_REG_CASE(22) PP_REG_CASE(23) PP_REG_CASE(24)
    default: return cudaErrorNotSupported;
  }
#undef PP_REG_CASE
  return cudaGetLastError();
}

cudaError_t launch_tridiag_factored(const Geometry& g, const DevTables& tb, int parts, bool trunc, cplx<double>* spec,
                                    const SideArgs& sd, cudaStream_t st) {
  if (parts == 1 && g.ny <= kScan64Rows && tb.tri_d.nsys <= kScan64Systems) {
    SideArgs side = sd;
    size_t smem = (size_t)((g.ny + 7) / 8) * 64 * 24;
    cudaError_t e = prepare_side<double>(g, side, 64, smem, spec, st);
    if (e != cudaSuccess) return e;
    if ((e = prep(k_tridiag_scan64, smem)) != cudaSuccess) return e;
    const int blocks = (g.nz * g.pitch + 7) / 8;
    k_tridiag_scan64<<<side.n + blocks, 64, smem, st>>>(g, tb.d.c, tb.tri_d, spec, side);
    return cudaGetLastError();
  }
  return launch_factored<double, true>(g, tb.d.a, tb.d.c, tb.tri_d, parts, -1, trunc, spec, sd, st);
}

cudaError_t launch_tridiag_factored_f32(const Geometry& g, const DevTables& tb, int parts, int low_modes, bool trunc,
                                        cplx<float>* spec, const SideArgs& sd, cudaStream_t st) {
  return launch_factored<float, false>(g, tb.f.a, tb.f.c, tb.tri_f, parts, low_modes, trunc, spec, sd, st);
}

}  // namespace pp
