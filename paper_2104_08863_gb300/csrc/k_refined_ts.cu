// The FP64-accurate timestep on FP32 units (the refined form of the projection timestep).
//
// The state (u, v, w) is carried through the step as FP32 pairs (hi, lo) with hi + lo equal to
// the FP64 value to about 2^-47 (same bytes as FP64), and every per-point operation runs in
// double-float arithmetic on the FP32 pipes (GB300 issues ~2 FP64 instructions per clock per SM
// against 128 FP32):
//   k_to_pairs        FP64 field -> pairs, in place (integer split, no FP64 instruction), and
//   k_from_pairs      back (faithful integer assembly);
//   k_momentum_df     one Heun stage (Eqs. 5-6) of the momentum right-hand side, the same
//                     central differences and edge-flux sharing as k_momentum, in double-float;
//   k_divergence_df   f = D(u*)/dt (Eq. 7) from the pairs, assembled as FP64 for the refined
//                     Poisson solve;
//   k_gradient_pairs  u = u* - dt G p (Eq. 4) from the pairs and the solve's FP32 pressure pair,
//                     FP64 out.
#include "df2.cuh"
#include "fpconv.cuh"
#include "internal.h"

namespace pp {

namespace {

__device__ __forceinline__ df dadd(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ df dsub(df a, df b) { return df_add(a, df_neg(b)); }
__device__ __forceinline__ df dmul(df a, df b) { return df_mul(a, b); }
__device__ __forceinline__ df dfma(df a, df b, df c) { return df_add(df_mul(a, b), c); }
__device__ __forceinline__ df dtwice(df a) { return df{2.f * a.hi, 2.f * a.lo}; }
// Sum of two pairs left unnormalised (TwoSum of the high parts, the low parts added): a valid
// double-float operand for a product, three operations cheaper than dadd.
__device__ __forceinline__ df uadd(df a, df b) {
  const df s = two_sum_df(a.hi, b.hi);
  return df{s.hi, s.lo + (a.lo + b.lo)};
}
__device__ __forceinline__ df usub(df a, df b) {
  const df s = two_diff_df(a.hi, b.hi);
  return df{s.hi, s.lo + (a.lo - b.lo)};
}
// Compensated accumulator (S, C) += c * x: the product's rounding error by FMAs, the sum's by
// TwoSum, all error terms collected in C (the Dot2 scheme); normalised once at the end.
struct Acc { float S, C; };
__device__ __forceinline__ void acc_prod(Acc& a, df c, df x) {
  const float p = c.hi * x.hi;
  float e = fmaf(c.hi, x.hi, -p);
  e = fmaf(c.hi, x.lo, e);
  e = fmaf(c.lo, x.hi, e);
  const df t = two_sum_df(a.S, p);
  a.S = t.hi;
  a.C += t.lo + e;
}
__device__ __forceinline__ Acc acc_of(df x) { return Acc{x.hi, x.lo}; }
__device__ __forceinline__ float2 acc_out(const Acc& a) {
  const df r = quick_two_sum_df(a.S, a.C);
  return make_float2(r.hi, r.lo);
}
__device__ __forceinline__ df ldp(const float2* p) {
  const float2 v = __ldg(p);
  return df{v.x, v.y};
}
__device__ __forceinline__ df split(double x) {
  df r;
  f64_split(x, r.hi, r.lo);
  return r;
}
__device__ __forceinline__ float2 f2(df a) { return make_float2(a.hi, a.lo); }

// The same operations on two values at once (df2.cuh): lane x one value, lane y the other, each
// lane giving the scalar form's result.
__device__ __forceinline__ df2 pk(df a, df b) { return df2{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)}; }
__device__ __forceinline__ df2 bc(df a) { return pk(a, a); }
__device__ __forceinline__ df2 uadd2(df2 a, df2 b) {
  const df2 s = two_sum2(a.hi, b.hi);
  return df2{s.hi, f2add(s.lo, f2add(a.lo, b.lo))};
}
__device__ __forceinline__ df2 usub2(df2 a, df2 b) {
  const df2 s = two_diff2(a.hi, b.hi);
  return df2{s.hi, f2add(s.lo, f2sub(a.lo, b.lo))};
}
__device__ __forceinline__ df2 dmul2(df2 a, df2 b) {
  const float2 p = f2mul(a.hi, b.hi);
  float2 e = f2fma(a.hi, b.hi, make_float2(-p.x, -p.y));
  e = f2fma(a.hi, b.lo, e);
  e = f2fma(a.lo, b.hi, e);
  return df2{p, e};
}
__device__ __forceinline__ df2 dtwice2(df2 a) {
  return df2{f2mul(a.hi, make_float2(2.f, 2.f)), f2mul(a.lo, make_float2(2.f, 2.f))};
}
struct Acc2 { float2 S, C; };
__device__ __forceinline__ void acc_prod2(Acc2& a, df2 c, df2 x) {
  const float2 p = f2mul(c.hi, x.hi);
  float2 e = f2fma(c.hi, x.hi, make_float2(-p.x, -p.y));
  e = f2fma(c.hi, x.lo, e);
  e = f2fma(c.lo, x.hi, e);
  const df2 t = two_sum2(a.S, p);
  a.S = t.hi;
  a.C = f2add(a.C, f2add(t.lo, e));
}
// (S + C) normalised (quick TwoSum) lane by lane; lane x as the first pair, lane y the second.
__device__ __forceinline__ void acc_out2(const Acc2& a, float2& x, float2& y) {
  const float2 s = f2add(a.S, a.C);
  const float2 lo = f2sub(a.C, f2sub(s, a.S));
  x = make_float2(s.x, lo.x);
  y = make_float2(s.y, lo.y);
}

constexpr int MTX = 32, MTZ = 8;

// Stage constants split on the host: the FP64 divisions of every thread took 10 % of the stage
// (512x384x512: 2.74 / 3.40 ms with them, 2.47 / 3.10 without).
struct MomCoefDF {
  double cdx, cdz, bdtnu;
  df cDx, cDz, cAx, cAz, fterm, alpha;
};

struct RowCoefDF {
  df c0, ca, cc, cay;
  df v0, va, vc, vay;
};

// Two values (16 bytes) per thread and step, the velocity triple in one launch (field blockIdx.y; its
// length is even): 740 us at 512x384x512 (6.5 TB/s), one value per step and a launch per field 865.
struct Triple {
  double* x[3];
  size_t n[3];
};

__global__ void __launch_bounds__(256) k_to_pairs(Triple f) {
  double* x = f.x[blockIdx.y];
  const size_t n2 = f.n[blockIdx.y] / 2, step = (size_t)gridDim.x * blockDim.x;
#pragma unroll 4
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += step) {
    const double2 v = reinterpret_cast<const double2*>(x)[i];
    const df p = split(v.x), q = split(v.y);
    reinterpret_cast<float4*>(x)[i] = make_float4(p.hi, p.lo, q.hi, q.lo);
  }
}

__global__ void __launch_bounds__(256) k_from_pairs(Triple f) {
  double* x = f.x[blockIdx.y];
  const size_t n2 = f.n[blockIdx.y] / 2, step = (size_t)gridDim.x * blockDim.x;
#pragma unroll 4
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += step) {
    const float4 v = reinterpret_cast<const float4*>(x)[i];
    reinterpret_cast<double2*>(x)[i] = make_double2(f32_add_to_f64(v.x, v.y), f32_add_to_f64(v.z, v.w));
  }
}

// out = alpha * base + beta * s + bdt * R(s) on pairs (see k_momentum for the stencil).
__global__ void __launch_bounds__(MTX * MTZ) k_momentum_df(Geometry g, MomArgsDF a, MomCoefDF mc,
                                                          const double* __restrict__ inv_dy,
                                                          const double* __restrict__ inv_h,
                                                          const double* __restrict__ lo,
                                                          const double* __restrict__ up, int jc) {
  extern __shared__ unsigned char smem_raw[];
  RowCoefDF* rc = reinterpret_cast<RowCoefDF*>(smem_raw);
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int j0 = blockIdx.z * jc;
  const int j1 = min(ny, j0 + jc);
  const double bdtnu = mc.bdtnu, cdx = mc.cdx, cdz = mc.cdz;
  for (int r = threadIdx.y * MTX + threadIdx.x; r < j1 - j0; r += MTX * MTZ) {
    const int j = j0 + r;
    RowCoefDF c;
    const double A = j > 0 ? lo[j] : 2.0 * inv_dy[0] * inv_dy[0];
    const double C = j < ny - 1 ? up[j] : 2.0 * inv_dy[ny - 1] * inv_dy[ny - 1];
    c.c0 = split(a.beta - 2.0 * cdx - 2.0 * cdz - bdtnu * (A + C));
    c.ca = split(j > 0 ? bdtnu * lo[j] : 0.0);
    c.cc = split(j < ny - 1 ? bdtnu * up[j] : 0.0);
    c.cay = split(-0.25 * a.bdt * inv_dy[j]);
    if (j >= 1) {
      const double va = bdtnu * inv_h[j] * inv_dy[j - 1], vc = bdtnu * inv_h[j] * inv_dy[j];
      c.v0 = split(a.beta - 2.0 * cdx - 2.0 * cdz - va - vc);
      c.va = split(va);
      c.vc = split(vc);
      c.vay = split(-0.25 * a.bdt * inv_h[j]);
    } else {
      c.v0 = c.va = c.vc = c.vay = df{0.f, 0.f};
    }
    rc[r] = c;
  }
  __syncthreads();
  const int i = blockIdx.x * MTX + threadIdx.x;
  const int k = blockIdx.y * MTZ + threadIdx.y;
  if (i >= nx || k >= nz) return;
  const df cDx = mc.cDx, cDz = mc.cDz, cAx = mc.cAx, cAz = mc.cAz;
  const df2 cD_xz = pk(cDx, cDz), cD_zx = pk(cDz, cDx), cA_xz = pk(cAx, cAz), cA_zx = pk(cAz, cAx);
  const df fterm = mc.fterm, alpha = mc.alpha;
  const bool has_base = a.bu != nullptr;
  const size_t plane = (size_t)nz * nx;
  const int im = i == 0 ? nx - 1 : i - 1, ip = i == nx - 1 ? 0 : i + 1;
  const int km = k == 0 ? nz - 1 : k - 1, kp = k == nz - 1 ? 0 : k + 1;
  const size_t oc = (size_t)k * nx + i, oxm = (size_t)k * nx + im, oxp = (size_t)k * nx + ip;
  const size_t ozm = (size_t)km * nx + i, ozp = (size_t)kp * nx + i;
  const size_t ozm_xp = (size_t)km * nx + ip, ozp_xm = (size_t)kp * nx + im;
  const float2* su = a.su;
  const float2* sv = a.sv;
  const float2* sw = a.sw;
  const df zero{0.f, 0.f};

  df u_m = zero, w_m = zero;
  df u_c = ldp(su + (size_t)j0 * plane + oc), w_c = ldp(sw + (size_t)j0 * plane + oc);
  df v_m = j0 > 0 ? ldp(sv + (size_t)(j0 - 1) * plane + oc) : zero;
  df v_c = ldp(sv + (size_t)j0 * plane + oc);
  df u_m_xp = zero, w_m_zp = zero;
  df e_uv = zero, e_vw = zero;
  if (j0 > 0) {
    const size_t pm = (size_t)(j0 - 1) * plane, pc = (size_t)j0 * plane;
    u_m = ldp(su + pm + oc);
    w_m = ldp(sw + pm + oc);
    u_m_xp = ldp(su + pm + oxp);
    w_m_zp = ldp(sw + pm + ozp);
    e_uv = dmul(uadd(ldp(sv + pc + oxm), v_c), uadd(u_m, u_c));
    e_vw = dmul(uadd(ldp(sv + pc + ozm), v_c), uadd(w_m, w_c));
  }
  df vs_m = uadd(v_m, v_c);
  if (j0 == 0) a.ov[oc] = has_base ? a.bv[oc] : f2(v_c);
  for (int j = j0; j < j1; ++j) {
    const RowCoefDF c = rc[j - j0];
    const size_t pc = (size_t)j * plane, pn = pc + plane;
    const bool top = j + 1 < ny;
    const df u_n = top ? ldp(su + pn + oc) : zero;
    const df w_n = top ? ldp(sw + pn + oc) : zero;
    const df v_n = ldp(sv + pn + oc);
    const df u_xm = ldp(su + pc + oxm), u_xp = ldp(su + pc + oxp), u_zm = ldp(su + pc + ozm), u_zp = ldp(su + pc + ozp);
    const df u_zm_xp = ldp(su + pc + ozm_xp);
    const df w_xm = ldp(sw + pc + oxm), w_xp = ldp(sw + pc + oxp), w_zm = ldp(sw + pc + ozm), w_zp = ldp(sw + pc + ozp);
    const df w_zp_xm = ldp(sw + pc + ozp_xm);
    const df v_xm = ldp(sv + pc + oxm), v_xp = ldp(sv + pc + oxp), v_zm = ldp(sv + pc + ozm), v_zp = ldp(sv + pc + ozp);
    df e_uv_n = zero, e_vw_n = zero;   // fluxes through face j+1 (zero on the top wall), as a pair
    if (top) {
      const df2 e = dmul2(uadd2(pk(ldp(sv + pn + oxm), ldp(sv + pn + ozm)), bc(v_n)), uadd2(pk(u_c, w_c), pk(u_n, w_n)));
      e_uv_n = df{e.hi.x, e.lo.x};
      e_vw_n = df{e.hi.y, e.lo.y};
    }
    const df e_uw = dmul(uadd(w_xm, w_c), uadd(u_zm, u_c));
    float2 bu2 = make_float2(0.f, 0.f), bw2 = bu2, bv2 = bu2;
    if (has_base) {   // the stage-2 base values, loaded together with the stencil
      bu2 = a.bu[pc + oc];
      bw2 = a.bw[pc + oc];
      if (j >= 1) bv2 = a.bv[pc + oc];
    }
    {   // u (lane x) and w (lane y): their equations mirror each other under x <-> z, term by term
      Acc2 acc{make_float2(fterm.hi, 0.f), make_float2(fterm.lo, 0.f)};
      if (has_base) acc_prod2(acc, bc(alpha), pk(df{bu2.x, bu2.y}, df{bw2.x, bw2.y}));
      const df2 cuw = pk(u_c, w_c);
      acc_prod2(acc, bc(c.c0), cuw);
      const df2 xp = pk(u_xp, w_zp), xm = pk(u_xm, w_zm);   // along x for u, along z for w
      const df2 s1 = uadd2(xp, xm);
      acc_prod2(acc, cD_xz, s1);
      acc_prod2(acc, cA_xz, dmul2(usub2(xp, xm), uadd2(s1, dtwice2(cuw))));
      acc_prod2(acc, cD_zx, uadd2(pk(u_zp, w_xp), pk(u_zm, w_xm)));
      acc_prod2(acc, cA_zx, usub2(dmul2(uadd2(pk(w_zp_xm, w_c), pk(w_zp, w_xp)), uadd2(pk(u_c, u_zm_xp), pk(u_zp, u_xp))),
                                  bc(e_uw)));
      acc_prod2(acc, bc(c.cay), usub2(pk(e_uv_n, e_vw_n), pk(e_uv, e_vw)));
      acc_prod2(acc, bc(c.ca), pk(u_m, w_m));
      acc_prod2(acc, bc(c.cc), pk(u_n, w_n));
      float2 ou, ow;
      acc_out2(acc, ou, ow);
      a.ou[pc + oc] = ou;
      a.ow[pc + oc] = ow;
    }
    if (j >= 1) {   // v at face j
      Acc acc{0.f, 0.f};
      if (has_base) acc_prod(acc, alpha, df{bv2.x, bv2.y});
      acc_prod(acc, c.v0, v_c);
      const df vs = uadd(v_c, v_n);
      acc_prod(acc, c.vay, dmul(usub(vs, vs_m), uadd(vs, vs_m)));
      acc_prod(acc, cDx, uadd(v_xp, v_xm));
      acc_prod(acc, cAx, usub(dmul(uadd(v_c, v_xp), uadd(u_m_xp, u_xp)), e_uv));
      acc_prod(acc, cDz, uadd(v_zp, v_zm));
      acc_prod(acc, cAz, usub(dmul(uadd(v_c, v_zp), uadd(w_m_zp, w_zp)), e_vw));
      acc_prod(acc, c.va, v_m);
      acc_prod(acc, c.vc, v_n);
      a.ov[pc + oc] = acc_out(acc);
    }
    vs_m = uadd(v_c, v_n);
    u_m = u_c; u_c = u_n;
    w_m = w_c; w_c = w_n;
    v_m = v_c; v_c = v_n;
    u_m_xp = u_xp;
    w_m_zp = w_zp;
    e_uv = e_uv_n;
    e_vw = e_vw_n;
  }
  if (j1 == ny) {
    const size_t pw = (size_t)ny * plane + oc;
    a.ov[pw] = has_base ? a.bv[pw] : __ldg(sv + pw);
  }
}

__device__ __forceinline__ df at0(float4 v) { return df{v.x, v.y}; }
__device__ __forceinline__ df at1(float4 v) { return df{v.z, v.w}; }
__device__ __forceinline__ float4 ld4(const float2* p) { return *reinterpret_cast<const float4*>(p); }

// f = D(u*) / dt at every cell from the pairs, written as FP64 (faithful assembly).  A thread takes
// two adjacent cells of a line, every field as 16-byte loads of two pairs, all in flight before the
// first use; 1/(dt dx) and 1/(dt dz) come split from the host (HBM-bound: 32 bytes per point;
// 512x384x512 620 us (5.2 TB/s), one cell per
// thread with divisions on the device 770).
__global__ void __launch_bounds__(256) k_divergence_df(Geometry g, const float2* __restrict__ u,
                                                      const float2* __restrict__ v, const float2* __restrict__ w,
                                                      const double* __restrict__ inv_dy, df cx, df cz, df cdt,
                                                      double* __restrict__ f) {
  const size_t plane = (size_t)g.nz * g.nx;
  const int line = blockIdx.x * blockDim.y + threadIdx.y;
  if (line >= g.ny * g.nz) return;
  const int j = line / g.nz, k = line - j * g.nz;
  const df cy = dmul(cdt, split(inv_dy[j]));
  const ptrdiff_t dzp = k + 1 == g.nz ? (ptrdiff_t)g.nx - (ptrdiff_t)plane : g.nx;
  for (int i0 = 2 * threadIdx.x; i0 < g.nx; i0 += 2 * blockDim.x) {
    const size_t idx = (size_t)line * g.nx + i0;
    const float4 uc = ld4(u + idx), wc = ld4(w + idx), wp = ld4(w + idx + dzp), vc = ld4(v + idx), vp = ld4(v + idx + plane);
    const df u2 = ldp(u + idx + (i0 + 2 == g.nx ? -(ptrdiff_t)i0 : 2));
    auto cell = [&](df ul, df ur, df wl, df wr, df vl, df vr) {
      df s = dmul(cx, dsub(ur, ul));
      s = dfma(cz, dsub(wr, wl), s);
      s = dfma(cy, dsub(vr, vl), s);
      return f32_add_to_f64(s.hi, s.lo);
    };
    *reinterpret_cast<double2*>(f + idx) = make_double2(cell(at0(uc), at1(uc), at0(wc), at0(wp), at0(vc), at0(vp)),
                                                        cell(at1(uc), u2, at1(wc), at1(wp), at1(vc), at1(vp)));
  }
}

// u = u* - dt G p (Eq. 4): u* as pairs, p = hi + lo the refined solve's FP32 pair, the result in
// FP64 (v's walls copied); the pressure differences and the products run in double-float and the
// sums are assembled into FP64 with integer operations (one FP64 addition per value).  p_out, when
// given, receives p in FP64.  Two adjacent cells per thread as above (HBM-bound: 64 bytes per point
// with p_out; 512x384x512 1.21 ms (5.3 TB/s), before 1.60).
__global__ void __launch_bounds__(256) k_gradient_pairs(Geometry g, const float* __restrict__ hi,
                                                        const float* __restrict__ lo, double* __restrict__ u,
                                                        double* __restrict__ v, double* __restrict__ w,
                                                        double* __restrict__ p_out, const double* __restrict__ inv_h,
                                                        df cx, df cz, df cdt) {
  const size_t plane = (size_t)g.nz * g.nx;
  const int line = blockIdx.x * blockDim.y + threadIdx.y;
  if (line >= (g.ny + 1) * g.nz) return;
  const int j = line / g.nz, k = line - j * g.nz;
  const bool cell = j < g.ny, inner = j >= 1 && cell;
  const df cy = inner ? dmul(cdt, split(inv_h[j])) : df{0.f, 0.f};
  const ptrdiff_t dzm = k == 0 ? (ptrdiff_t)plane - g.nx : -(ptrdiff_t)g.nx;
  auto P2 = [&](size_t o) {   // the pressure pairs of two cells
    const float2 h = __ldg(reinterpret_cast<const float2*>(hi + o)), l = __ldg(reinterpret_cast<const float2*>(lo + o));
    return make_float4(h.x, l.x, h.y, l.y);
  };
  auto out = [](df a, df b) { return make_double2(f32_add_to_f64(a.hi, a.lo), f32_add_to_f64(b.hi, b.lo)); };
  for (int i0 = 2 * threadIdx.x; i0 < g.nx; i0 += 2 * blockDim.x) {
    const size_t idx = (size_t)line * g.nx + i0;
    const float4 vv = *reinterpret_cast<const float4*>(v + idx);
    df v0 = at0(vv), v1 = at1(vv);
    if (cell) {
      const float4 uu = *reinterpret_cast<const float4*>(u + idx), ww = *reinterpret_cast<const float4*>(w + idx);
      const float4 pc = P2(idx), pz = P2(idx + dzm), py = inner ? P2(idx - plane) : pc;
      const size_t ox = idx + (i0 == 0 ? g.nx - 1 : -1);
      const df pl{__ldg(hi + ox), __ldg(lo + ox)};
      *reinterpret_cast<double2*>(u + idx) = out(dsub(at0(uu), dmul(cx, dsub(at0(pc), pl))),
                                                 dsub(at1(uu), dmul(cx, dsub(at1(pc), at0(pc)))));
      *reinterpret_cast<double2*>(w + idx) = out(dsub(at0(ww), dmul(cz, dsub(at0(pc), at0(pz)))),
                                                 dsub(at1(ww), dmul(cz, dsub(at1(pc), at1(pz)))));
      if (p_out) *reinterpret_cast<double2*>(p_out + idx) = out(at0(pc), at1(pc));
      if (inner) {
        v0 = dsub(v0, dmul(cy, dsub(at0(pc), at0(py))));
        v1 = dsub(v1, dmul(cy, dsub(at1(pc), at1(py))));
      }
    }
    *reinterpret_cast<double2*>(v + idx) = out(v0, v1);
  }
}

// CTAs of tx pairs of cells by 256 / tx lines.
struct LineTiles { dim3 grid, block; };
LineTiles pair_tiles(const Geometry& g, int nlines) {
  const int tx = g.nx / 2 < 256 ? g.nx / 2 : 256, ty = 256 / tx;
  return LineTiles{dim3((nlines + ty - 1) / ty), dim3(tx, ty)};
}

df split_host(double x) {
  df r;
  f64_split(x, r.hi, r.lo);
  return r;
}

// Grid of the in-place conversions: 16 CTAs per SM, each field of the triple in its own rows.
dim3 triple_grid(const Triple& f) {
  const size_t most = f.n[0] > f.n[1] ? f.n[0] : f.n[1], blocks = (most / 2 + 255) / 256;
  return dim3((unsigned)(blocks < 152 * 16 ? (blocks ? blocks : 1) : 152 * 16), 3);
}
Triple triple(const Geometry& g, double* u, double* v, double* w) {
  const size_t plane = (size_t)g.nz * g.nx;
  return Triple{{u, v, w}, {plane * g.ny, plane * (g.ny + 1), plane * g.ny}};
}

}  // namespace

cudaError_t launch_to_pairs(const Geometry& g, double* u, double* v, double* w, cudaStream_t st) {
  const Triple f = triple(g, u, v, w);
  k_to_pairs<<<triple_grid(f), 256, 0, st>>>(f);
  return cudaGetLastError();
}

cudaError_t launch_from_pairs(const Geometry& g, double* u, double* v, double* w, cudaStream_t st) {
  const Triple f = triple(g, u, v, w);
  k_from_pairs<<<triple_grid(f), 256, 0, st>>>(f);
  return cudaGetLastError();
}

cudaError_t launch_momentum_df(const Geometry& g, const DevTables& tb, const MomArgsDF& a, cudaStream_t st) {
  const int tx = (g.nx + MTX - 1) / MTX, tz = (g.nz + MTZ - 1) / MTZ;
  const long long tiles = (long long)tx * tz;
  const int jc = momentum_chunk_rows(tiles, g.ny), chunks = (g.ny + jc - 1) / jc;
  const size_t smem = sizeof(RowCoefDF) * (size_t)jc;
  const cudaError_t e = ensure_smem_limit((const void*)k_momentum_df, smem);
  if (e != cudaSuccess) return e;
  dim3 grid(tx, tz, chunks), block(MTX, MTZ);
  const double bdtnu = a.bdt * a.nu, cdx = bdtnu / (g.dx * g.dx), cdz = bdtnu / (g.dz * g.dz);
  const MomCoefDF mc{cdx, cdz, bdtnu, split_host(cdx), split_host(cdz), split_host(-0.25 * a.bdt / g.dx),
                     split_host(-0.25 * a.bdt / g.dz), split_host(a.bdt * a.fx), split_host(a.alpha)};
  k_momentum_df<<<grid, block, smem, st>>>(g, a, mc, tb.d.inv_dy, tb.d.inv_h, tb.d.a, tb.d.c, jc);
  return cudaGetLastError();
}

cudaError_t launch_divergence_df(const Geometry& g, const DevTables& tb, const float2* u, const float2* v,
                                 const float2* w, double dt, double* f, cudaStream_t st) {
  const LineTiles t = pair_tiles(g, g.ny * g.nz);
  const double inv_dt = 1.0 / dt;
  k_divergence_df<<<t.grid, t.block, 0, st>>>(g, u, v, w, tb.d.inv_dy, split_host(inv_dt / g.dx),
                                              split_host(inv_dt / g.dz), split_host(inv_dt), f);
  return cudaGetLastError();
}

cudaError_t launch_gradient_pairs(const Geometry& g, const DevTables& tb, const float* hi, const float* lo, double* u,
                                  double* v, double* w, double* p_out, double dt, cudaStream_t st) {
  const LineTiles t = pair_tiles(g, (g.ny + 1) * g.nz);
  k_gradient_pairs<<<t.grid, t.block, 0, st>>>(g, hi, lo, u, v, w, p_out, tb.d.inv_h, split_host(dt / g.dx),
                                               split_host(dt / g.dz), split_host(dt));
  return cudaGetLastError();
}

}  // namespace pp
