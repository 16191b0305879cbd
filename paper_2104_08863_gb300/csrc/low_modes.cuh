// The modes of a solve that run apart from the main wall-normal pass: the singular (0, 0) mode
// (compatibility and gauge) and, in the FP32 forms, the FP64 systems with kx <= L, |kz| <= L.  They are extra CTAs at the head of the main pass's grid, so their serial
// FP64 chains run beside its tiles instead of in launches of their own before and after it (a
// 192x96x192 refined adjoint spent 3 x 65 of 485 us there, a 256x192x256 FP32 projection with
// its gradient 2 x 73 of 733).
//
// A system is solved with the exact elimination (Thomas) whose pivots 1/beta_j depend only on
// the grid and are built once per plan in FP64 (k_low_setup, the cancellation-free margin
// recurrence).  With known pivots the two sweeps are first-order linear recurrences with
// coefficients in (0, 1),
//   g_j = -F_j + (a_j / beta_{j-1}) g_{j-1},     x_j = g_j / beta_j + (c_j / beta_j) x_{j+1},
// so a group of threads takes contiguous rows each, and the carries between them come from a scan
// of affine maps (shuffles in a warp, shared memory across the warps).  What bounds it is the
// FP64 latency of the ny / group dependent rows per sweep: 768 rows on 128 threads take 6 steps
// each way, where one warp per system with divisions on the chain took 93 us.  Up to 256 rows the
// group is one warp (at most 8 rows a lane).
#pragma once

#include "internal.h"

namespace pp {

constexpr int kLowMaxGroups = 2;   // systems per CTA at most
constexpr int kLowMaxWarps = 8;    // 128 threads each

// The threads that work on one system: nt of them (a multiple of 32), this one the t-th, with a
// named barrier and 3 nt / 32 doubles of shared memory of their own.
struct LowGroup {
  int t, nt, bar;
  double* red;
  // barriers 1 and 2 by name (a number in a register would reserve all sixteen for the kernel)
  __device__ __forceinline__ void sync() const {
    if (bar == 1) asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"r"(nt) : "memory");
  }
};

// Sum of N values over the group, in every thread.
template <int N>
__device__ __forceinline__ void low_sum(double (&v)[N], const LowGroup& gr) {
#pragma unroll
  for (int k = 0; k < N; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  const int nw = gr.nt >> 5;
  if (nw == 1) return;
  gr.sync();   // red is free again
  if ((gr.t & 31) == 0)
#pragma unroll
    for (int k = 0; k < N; ++k) gr.red[(gr.t >> 5) * N + k] = v[k];
  gr.sync();
#pragma unroll
  for (int k = 0; k < N; ++k) {
    double s = 0.0;
    for (int w = 0; w < nw; ++w) s += gr.red[w * N + k];
    v[k] = s;
  }
}

// The value that enters this thread's rows when thread t maps an incoming y to A y + B, applied
// in thread order (UP) or in reverse, with 0 before the first: a warp scan of the maps, then the
// maps of the group's other warps.
template <bool UP>
__device__ __forceinline__ double2 low_carry(double A, double2 B, const LowGroup& gr) {
  const int lane = gr.t & 31, warp = gr.t >> 5, nw = gr.nt >> 5;
  double* red = gr.red;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double Ap = UP ? __shfl_up_sync(0xffffffffu, A, d) : __shfl_down_sync(0xffffffffu, A, d);
    const double Bx = UP ? __shfl_up_sync(0xffffffffu, B.x, d) : __shfl_down_sync(0xffffffffu, B.x, d);
    const double By = UP ? __shfl_up_sync(0xffffffffu, B.y, d) : __shfl_down_sync(0xffffffffu, B.y, d);
    if (UP ? lane >= d : lane + d < 32) {
      B = make_double2(fma(A, Bx, B.x), fma(A, By, B.y));
      A *= Ap;
    }
  }
  double2 in = make_double2(0.0, 0.0);   // carry into this warp
  if (nw > 1) {
    gr.sync();
    if (lane == (UP ? 31 : 0)) {
      red[3 * warp] = A;
      red[3 * warp + 1] = B.x;
      red[3 * warp + 2] = B.y;
    }
    gr.sync();
    for (int q = 0; q < nw - 1; ++q) {
      const int w = UP ? q : nw - 1 - q;
      if (UP ? w < warp : w > warp)
        in = make_double2(fma(red[3 * w], in.x, red[3 * w + 1]), fma(red[3 * w], in.y, red[3 * w + 2]));
    }
  }
  const double Ae = UP ? __shfl_up_sync(0xffffffffu, A, 1) : __shfl_down_sync(0xffffffffu, A, 1);
  const double Bx = UP ? __shfl_up_sync(0xffffffffu, B.x, 1) : __shfl_down_sync(0xffffffffu, B.x, 1);
  const double By = UP ? __shfl_up_sync(0xffffffffu, B.y, 1) : __shfl_down_sync(0xffffffffu, B.y, 1);
  if (lane == (UP ? 0 : 31)) return in;
  return make_double2(fma(Ae, in.x, Bx), fma(Ae, in.y, By));
}

// The (0, 0) mode: T p = F - mean with sum_j dy_j p_j = 0, by the exact flux prefix sums
// q_j = sum_{l<=j} dy_l F^c_l, p_0 = 0, p_{j+1} = p_j + h_{j+1} q_j, then the removal of the
// dy-weighted mean.  y holds ny values.
template <typename TD>
__device__ __forceinline__ void low_mode00(const Geometry& g, const SideArgs& sd, cplx<TD>* __restrict__ spec,
                                           double2* y, const LowGroup& gr, int lo, int hi) {
  const double* dy = sd.dy;
  const double* h = sd.h;
  const int ny = g.ny, gauge = sd.gauge;
  double* acc = sd.acc;
  const size_t rstride = (size_t)g.nz * g.pitch;
  double s[3] = {0.0, 0.0, 0.0};
#pragma unroll 4
  for (int j = lo; j < hi; ++j) {
    const cplx<TD> F = ld_c(spec + (size_t)j * rstride);
    y[j] = make_double2(double(F.x), double(F.y));
    s[0] = fma(__ldg(dy + j), y[j].x, s[0]);
    s[1] = fma(__ldg(dy + j), y[j].y, s[1]);
    s[2] += __ldg(dy + j);
  }
  low_sum<3>(s, gr);
  const double sw = s[2], mr = s[0] / sw, mi = s[1] / sw;
  // <f> = (sum_j dy_j F_j) / (sum_j dy_j Nx Nz): kept for the residual of the refined solve
  if (gauge == GAUGE_STORE_MEAN && gr.t == 0) acc[0] = mr / ((double)g.nx * (double)g.nz);
  double2 q = make_double2(0.0, 0.0);   // flux sums of the thread's rows
#pragma unroll 4
  for (int j = lo; j < hi; ++j) {
    q = make_double2(fma(__ldg(dy + j), y[j].x - mr, q.x), fma(__ldg(dy + j), y[j].y - mi, q.y));
    y[j] = q;
  }
  const double2 q0 = low_carry<true>(1.0, q, gr);
  double2 p = make_double2(0.0, 0.0);   // pressure sums, exclusive of row j
#pragma unroll 4
  for (int j = lo; j < hi; ++j) {
    const double hj = j + 1 < ny ? __ldg(h + j + 1) : 0.0;
    const double2 t = make_double2(y[j].x + q0.x, y[j].y + q0.y);
    y[j] = p;
    p = make_double2(fma(hj, t.x, p.x), fma(hj, t.y, p.y));
  }
  const double2 p0 = low_carry<true>(1.0, p, gr);
  double m[2] = {0.0, 0.0};
#pragma unroll 4
  for (int j = lo; j < hi; ++j) {
    y[j] = make_double2(y[j].x + p0.x, y[j].y + p0.y);
    m[0] = fma(__ldg(dy + j), y[j].x, m[0]);
    m[1] = fma(__ldg(dy + j), y[j].y, m[1]);
  }
  low_sum<2>(m, gr);
  double m0 = m[0] / sw;
  const double m1 = m[1] / sw;
  // Offset gauge: the running total p has weighted sum acc[1]; shift this (0, 0) profile by
  // -acc[1] / sum(dy) so that sum_j dy_j (P_j + shift) = -acc[1].
  if (gauge == GAUGE_OFFSET) m0 += acc[1] / sw;
#pragma unroll 4
  for (int j = lo; j < hi; ++j)
    st_c(spec + (size_t)j * rstride, mk<TD>(TD(y[j].x - m0), TD(y[j].y - m1)));
}

// The systems blk * per .. of the list (kx = sys mod (L+1), then kz = 0..L, -L..-1; sys = 0 the
// (0, 0) mode), a group of the CTA's threads to each; the CTA's dynamic shared memory holds 16 ny
// bytes per group.  A function of its own: its FP64 state does not raise the registers of the
// kernel whose grid it shares, and all heights of the FP32 kernels run the same code (64 solves
// of mixed heights in turn: 2450 us inlined, 2390).  The coefficients go through the read-only
// path, which lets the unrolled loops load them ahead of their chains and their stores.
template <typename TD>
__device__ __noinline__ void low_system(const Geometry& g, const SideArgs& sd, cplx<TD>* __restrict__ spec, int blk) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[3 * kLowMaxWarps];
  const int group = (int)threadIdx.x / sd.threads;
  const int sys = blk * sd.per + group;
  if (group >= sd.per || sys >= sd.nsys) return;
  const LowGroup gr{(int)threadIdx.x - group * sd.threads, sd.threads, 1 + group, red + 3 * group * (sd.threads >> 5)};
  const int ny = g.ny, ch = (ny + gr.nt - 1) / gr.nt;
  double2* y = reinterpret_cast<double2*>(smem_raw) + (size_t)group * ny;   // every thread touches its own rows only
  const int lo = min(ny, gr.t * ch), hi = min(ny, lo + ch);
  if (sys == 0) {
    low_mode00<TD>(g, sd, spec, y, gr, lo, hi);
    return;
  }
  const int kx = sys % (sd.low + 1), q = sys / (sd.low + 1);
  const int kz = q <= sd.low ? q : g.nz - (q - sd.low);
  const size_t rstride = (size_t)g.nz * g.pitch;
  cplx<TD>* col = spec + (size_t)kz * g.pitch + kx;
  const double* ta = sd.a;
  const double* tc = sd.c;
  const double* rb = sd.rb + (size_t)sys * ny;
  double A = 1.0;
  double2 B = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int j = lo; j < hi; ++j) {
    const cplx<TD> F = ld_c(col + (size_t)j * rstride);
    const double mult = j > 0 ? __ldg(ta + j) * __ldg(rb + j - 1) : 0.0;
    B = make_double2(fma(mult, B.x, -double(F.x)), fma(mult, B.y, -double(F.y)));
    A *= mult;
    y[j] = B;
  }
  const double2 gin = low_carry<true>(A, B, gr);
  double Pm = 1.0;
#pragma unroll 4
  for (int j = lo; j < hi; ++j) {
    Pm *= j > 0 ? __ldg(ta + j) * __ldg(rb + j - 1) : 0.0;
    y[j] = make_double2(fma(Pm, gin.x, y[j].x), fma(Pm, gin.y, y[j].y));
  }
  A = 1.0;
  B = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int j = hi - 1; j >= lo; --j) {
    const double r = __ldg(rb + j), cr = __ldg(tc + j) * r;
    B = make_double2(fma(cr, B.x, r * y[j].x), fma(cr, B.y, r * y[j].y));
    A *= cr;
    y[j] = B;
  }
  const double2 xin = low_carry<false>(A, B, gr);
  double Q = 1.0;
#pragma unroll 4
  for (int j = hi - 1; j >= lo; --j) {
    Q *= __ldg(tc + j) * __ldg(rb + j);
    st_c(col + (size_t)j * rstride, mk<TD>(TD(fma(Q, xin.x, y[j].x)), TD(fma(Q, xin.y, y[j].y))));
  }
}

}  // namespace pp
