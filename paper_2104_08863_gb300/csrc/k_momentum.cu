// Momentum predictor of the fully explicit projection method (Sec. 2, Eqs. 3, 5, 6).
//
// One launch evaluates one stage of Heun's RK2 on the staggered faces:
//   out = alpha * base + beta * s + bdt * R(s),   R(s) = -N(s) + nu lap(s) + (fx, 0, 0)
// stage 1: (alpha, beta, bdt) = (0, 1, dt)       -> u_bar = u + dt R(u)
// stage 2: (alpha, beta, bdt) = (1/2, 1/2, dt/2) -> u_star = (u + u_bar + dt R(u_bar)) / 2
//                                                 = u + dt/2 (R(u) + R(u_bar))
// The advection N is the divergence form with two-point face averages: each flux through a
// face of a momentum control volume is the product of the two averaged velocities there, and the
// fluxes through the no-slip walls vanish.  The diffusion is the three-point Laplacian; the walls
// enter u and w through the wall value 0 half a cell from the first node.  v's wall faces are
// boundary values and are copied (stage 1) or left unchanged (stage 2, in place).
//
// Every flux is shared by two momentum equations: the u-v edge flux (x-face i, y-face f) is the
// y-flux of u and the x-flux of v, likewise u-w (z of u, x of w) and v-w (y of w, z of v).  A
// thread owns V adjacent x points of one k and marches up the rows of its chunk: the y-fluxes and
// the y-neighbours roll through registers, the x-neighbours inside the V points and the x-fluxes
// between them are the thread's own (V + 1 evaluations for V points), every field is read as
// 16-byte vectors (V = 4 FP32, 2 FP64) plus the two x-neighbours outside, z-neighbours through L1.
// Per-row coefficients (stretched y, no-slip wall rows, the stage factors) are built once per CTA
// in shared memory from the plan's FP64 metric tables.
//
// FP32 is bound by HBM (24 / 36 bytes per point) once the instructions are few enough: one point
// per thread issued 221 instructions per point, most of them addresses, at 20 warps per SM
// (269 / 372 us for the two stages of 384x192x256); now 113 / 131 us (4.0 / 5.2 TB/s).  FP64 is
// bound by its issue rate of two instructions per clock and SM (about 59 / 62 per point, before 67 / 70):
// 512x384x512 11.0 / 11.5 ms, before 12.6 / 12.5.
#include "internal.h"

namespace pp {

// Rows per chunk: the split of the rows that minimises (CTAs on the busiest SM) x (rows + the
// chunk's own start, worth about one row), so that small grids fill the SMs and large ones do not
// repeat the start; one chunk to four rows at most (5 or 9 rows: chunks of 3), at most 1024 rows to a
// chunk (64 KB of coefficients).  (64x64x64 FP64: 45 us per stage on 152 SMs, 88 us when chunks had at
// least 16 rows and filled 64 SMs.)
int momentum_chunk_rows(long long tiles, int rows) {
  int best = rows;
  double cost = -1.0;
  for (int chunks = (rows + 1023) / 1024; chunks <= (rows + 3) / 4; ++chunks) {
    const int jc = (rows + chunks - 1) / chunks;
    const long long ctas = tiles * ((rows + jc - 1) / jc);
    const double t = (double)((ctas + 151) / 152) * (jc + 1.0);
    if (cost < 0.0 || t < cost) {
      cost = t;
      best = jc;
    }
    if (ctas > 152LL * 64) break;
  }
  return best;
}

namespace {

constexpr int MOM_THREADS = 256;

template <typename T>
struct RowCoef {    // u and w rows j, v faces f = j
  T c0, ca, cc, cay;         // centre, j-1, j+1 diffusion weights; y-advection scale
  T v0, va, vc, vay;         // the same for v at face j (j = 1..ny-1)
};

// Stage constants, from the host (no FP64 division on the device).
struct MomCoef {
  double cdx, cdz, cax, caz, bdtnu, fterm;
};

template <typename T, int V> struct alignas(sizeof(T) * V) MVec { T x[V]; };
template <typename T, int V>
__device__ __forceinline__ MVec<T, V> vldg(const T* p) {
  MVec<T, V> r;
  if constexpr (sizeof(T) * V == 16 && sizeof(T) == 4) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p));
    r.x[0] = q.x; r.x[1] = q.y; r.x[2] = q.z; r.x[3] = q.w;
  } else if constexpr (sizeof(T) == 4) {
    const float2 q = __ldg(reinterpret_cast<const float2*>(p));
    r.x[0] = q.x; r.x[1] = q.y;
  } else {
    const double2 q = __ldg(reinterpret_cast<const double2*>(p));
    r.x[0] = q.x; r.x[1] = q.y;
  }
  return r;
}
template <typename T, int V>
__device__ __forceinline__ MVec<T, V> vldv(const T* p) { return *reinterpret_cast<const MVec<T, V>*>(p); }
template <typename T, int V>
__device__ __forceinline__ void vst(T* p, const MVec<T, V>& r) { *reinterpret_cast<MVec<T, V>*>(p) = r; }

// SHARE: the u-w and v-w fluxes through z-face k + 1 are those that the thread at k + 1 computes
// anyway, taken from it through shared memory (two buffers, one barrier per row) instead of computed
// again; the last line of a tile computes them.  Only the FP64 kernel does (7 of its 62 instructions
// per point go, 4 in two stay as differences): 512x384x512 11.44 / 11.94 -> 10.97 / 11.53 ms; FP32 is
// not bound by its arithmetic.
template <typename T, int V, bool BASE, bool SHARE>
__global__ void __launch_bounds__(MOM_THREADS, 2) k_momentum(Geometry g, MomArgs<T> a, MomCoef mc,
                                                            const double* __restrict__ inv_dy,
                                                            const double* __restrict__ inv_h,
                                                            const double* __restrict__ lo,
                                                            const double* __restrict__ up, int jlo, int jhi, int jc) {
  using Vt = MVec<T, V>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RowCoef<T>* rc = reinterpret_cast<RowCoef<T>*>(smem_raw);
  __shared__ MVec<T, V> edge[SHARE ? 2 : 1][SHARE ? 2 * MOM_THREADS : 1];   // [buffer][u-w, v-w][thread]
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  // the second stage begins with the rows that the first wrote last, while they are in the L2 (512x384x512
  // FP64: 11.55 -> 11.46 ms)
  const int j0 = jlo + (BASE ? gridDim.z - 1 - blockIdx.z : blockIdx.z) * jc;
  const int j1 = min(jhi, j0 + jc);
  for (int r = threadIdx.y * blockDim.x + threadIdx.x; r < j1 - j0; r += blockDim.x * blockDim.y) {
    const int j = j0 + r;
    RowCoef<T> c;
    const double A = j > 0 ? lo[j] : 2.0 * inv_dy[0] * inv_dy[0];
    const double C = j < ny - 1 ? up[j] : 2.0 * inv_dy[ny - 1] * inv_dy[ny - 1];
    c.c0 = T(a.beta - 2.0 * mc.cdx - 2.0 * mc.cdz - mc.bdtnu * (A + C));
    c.ca = T(j > 0 ? mc.bdtnu * lo[j] : 0.0);
    c.cc = T(j < ny - 1 ? mc.bdtnu * up[j] : 0.0);
    c.cay = T(-0.25 * a.bdt * inv_dy[j]);
    if (j >= 1) {
      const double va = mc.bdtnu * inv_h[j] * inv_dy[j - 1], vc = mc.bdtnu * inv_h[j] * inv_dy[j];
      c.v0 = T(a.beta - 2.0 * mc.cdx - 2.0 * mc.cdz - va - vc);
      c.va = T(va);
      c.vc = T(vc);
      c.vay = T(-0.25 * a.bdt * inv_h[j]);
    } else {
      c.v0 = c.va = c.vc = c.vay = T(0);
    }
    rc[r] = c;
  }
  __syncthreads();
  int i0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  int k = blockIdx.y * blockDim.y + threadIdx.y;
  const bool live = i0 < nx && k < nz;
  if (!live) {
    if constexpr (!SHARE) return;
    i0 = 0;   // takes part in the barriers with the source values of line 0, loading no base, storing nothing
    k = 0;
  }
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const bool shared_zp = SHARE && threadIdx.y + 1 < blockDim.y && k + 1 < nz && live;
  const T cDx = T(mc.cdx), cDz = T(mc.cdz), cAx = T(mc.cax), cAz = T(mc.caz);
  const T fterm = T(mc.fterm), alpha = T(a.alpha);
  const ptrdiff_t plane = (ptrdiff_t)nz * nx;
  // offsets from a point: the x-neighbours outside the V points, the z-neighbour lines (periodic)
  const ptrdiff_t dxm = i0 == 0 ? nx - 1 : -1, dxp = i0 + V == nx ? -i0 : V;
  const ptrdiff_t dzm = k == 0 ? plane - nx : -(ptrdiff_t)nx, dzp = k == nz - 1 ? nx - plane : nx;
  ptrdiff_t o = (ptrdiff_t)j0 * plane + (ptrdiff_t)k * nx + i0;   // row j of the chunk
  const T* su = a.su;
  const T* sv = a.sv;
  const T* sw = a.sw;

  // rolling state: rows j-1 and j, the fluxes through face j (zero on the wall)
  Vt u_m{}, w_m{}, v_m{}, wm_zp{};          // row j-1 (0 below the wall); w(j-1, k+1)
  Vt u_c = vldg<T, V>(su + o), w_c = vldg<T, V>(sw + o), v_c = vldg<T, V>(sv + o), v_zm = vldg<T, V>(sv + o + dzm);
  T u_xp = __ldg(su + o + dxp), v_xm = __ldg(sv + o + dxm), v_xp = __ldg(sv + o + dxp);
  T e_uv[V + 1], e_vw[V];                   // u-v at i0 .. i0 + V, v-w
#pragma unroll
  for (int q = 0; q < V; ++q) e_uv[q] = e_vw[q] = T(0);
  e_uv[V] = T(0);
  // u-v edge fluxes at i0 .. i0 + V from v and its x-neighbours on the face and u below and above
  auto uv_flux = [&](T vxm, const Vt& v, T vxp, const Vt& ua, T uaxp, const Vt& ub, T ubxp, T* e) {
#pragma unroll
    for (int q = 0; q <= V; ++q) {
      const T vs = (q ? v.x[q - 1] : vxm) + (q < V ? v.x[q] : vxp);
      const T us = q < V ? ua.x[q] + ub.x[q] : uaxp + ubxp;
      e[q] = vs * us;
    }
  };
  if (j0 > 0) {
    u_m = vldg<T, V>(su + o - plane);
    w_m = vldg<T, V>(sw + o - plane);
    v_m = vldg<T, V>(sv + o - plane);
    wm_zp = vldg<T, V>(sw + o - plane + dzp);
    uv_flux(v_xm, v_c, v_xp, u_m, __ldg(su + o - plane + dxp), u_c, u_xp, e_uv);
#pragma unroll
    for (int q = 0; q < V; ++q) e_vw[q] = (v_zm.x[q] + v_c.x[q]) * (w_m.x[q] + w_c.x[q]);
  } else {   // bottom wall face of v: boundary value
    if (live) vst<T, V>(a.ov + o, BASE ? vldv<T, V>(a.bv + o) : v_c);
  }
  for (int j = j0; j < j1; ++j, o += plane) {
    const RowCoef<T> c = rc[j - j0];
    const bool top = j + 1 < ny;
    // row j + 1 (zero above the top wall), then the neighbours in row j
    Vt u_n{}, w_n{};
    T un_xp = T(0);
    if (top) {
      u_n = vldg<T, V>(su + o + plane);
      w_n = vldg<T, V>(sw + o + plane);
      un_xp = __ldg(su + o + plane + dxp);
    }
    const Vt v_n = vldg<T, V>(sv + o + plane), vn_zm = vldg<T, V>(sv + o + plane + dzm);
    const T vn_xm = __ldg(sv + o + plane + dxm), vn_xp = __ldg(sv + o + plane + dxp);
    const Vt u_zm = vldg<T, V>(su + o + dzm), u_zp = vldg<T, V>(su + o + dzp);
    const Vt w_zm = vldg<T, V>(sw + o + dzm), w_zp = vldg<T, V>(sw + o + dzp), v_zp = vldg<T, V>(sv + o + dzp);
    const T u_xm = __ldg(su + o + dxm), uzm_xp = __ldg(su + o + dzm + dxp);
    const T w_xm = __ldg(sw + o + dxm), w_xp = __ldg(sw + o + dxp);
    T wzp_xm = T(0);
    if (!shared_zp) wzp_xm = __ldg(sw + o + dzp + dxm);
    Vt bu{}, bw{}, bv{};
    if (BASE && live) {   // (0, 0) has a thread of its own, which writes its result over the base in place
      bu = vldv<T, V>(a.bu + o);
      bw = vldv<T, V>(a.bw + o);
      bv = vldv<T, V>(a.bv + o);
    }
    // fluxes through face j+1 (zero on the top wall), and the u-w edge fluxes at i0 .. i0 + V
    T e_uv_n[V + 1], e_vw_n[V], e_uw[V + 1];
    if (top) {
      uv_flux(vn_xm, v_n, vn_xp, u_c, u_xp, u_n, un_xp, e_uv_n);
#pragma unroll
      for (int q = 0; q < V; ++q) e_vw_n[q] = (vn_zm.x[q] + v_n.x[q]) * (w_c.x[q] + w_n.x[q]);
    } else {
#pragma unroll
      for (int q = 0; q < V; ++q) e_uv_n[q] = e_vw_n[q] = T(0);
      e_uv_n[V] = T(0);
    }
    uv_flux(w_xm, w_c, w_xp, u_zm, uzm_xp, u_c, u_xp, e_uw);   // (w_xm + w_c) (u_zm + u_c)
    T fz_u[V], fz_v[V];   // flux differences across the cell in z: u-w for u, v-w for v
    if constexpr (SHARE) {
      Vt* e = edge[(j - j0) & 1];
      Vt su_, sv_;
#pragma unroll
      for (int q = 0; q < V; ++q) {
        su_.x[q] = e_uw[q];
        sv_.x[q] = e_vw[q];
      }
      e[tid] = su_;
      e[MOM_THREADS + tid] = sv_;
      __syncthreads();
      if (shared_zp) {
        const Vt nu_ = e[tid + blockDim.x], nv_ = e[MOM_THREADS + tid + blockDim.x];
#pragma unroll
        for (int q = 0; q < V; ++q) {
          fz_u[q] = nu_.x[q] - e_uw[q];
          fz_v[q] = nv_.x[q] - e_vw[q];
        }
      }
    }
    if (!shared_zp) {
      Vt wmz = wm_zp;   // w(j-1, k+1): rolled, or (few lines) loaded again
      if constexpr (SHARE) {
        if (j > j0) wmz = vldg<T, V>(sw + o - plane + dzp);
      }
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const T wzpxm = q ? w_zp.x[q - 1] : wzp_xm;
        fz_u[q] = (wzpxm + w_zp.x[q]) * (u_c.x[q] + u_zp.x[q]) - e_uw[q];
        fz_v[q] = (v_c.x[q] + v_zp.x[q]) * (wmz.x[q] + w_zp.x[q]) - e_vw[q];
      }
    }
    Vt ru, rw, rv;
#pragma unroll
    for (int q = 0; q < V; ++q) {
      const T uc = u_c.x[q], wc = w_c.x[q], vv = v_c.x[q];
      const T uxm = q ? u_c.x[q - 1] : u_xm, uxp = q + 1 < V ? u_c.x[q + 1] : u_xp;
      const T wxm = q ? w_c.x[q - 1] : w_xm, wxp = q + 1 < V ? w_c.x[q + 1] : w_xp;
      const T vxm = q ? v_c.x[q - 1] : v_xm, vxp = q + 1 < V ? v_c.x[q + 1] : v_xp;
      {   // u
        T acc = fterm;
        if constexpr (BASE) acc = alpha * bu.x[q] + acc;
        acc = c.c0 * uc + acc;
        const T sx = uxp + uxm;
        acc = cDx * sx + acc;
        acc = cAx * ((uxp - uxm) * (sx + T(2) * uc)) + acc;
        acc = cDz * (u_zp.x[q] + u_zm.x[q]) + acc;
        acc = cAz * fz_u[q] + acc;
        acc = c.cay * (e_uv_n[q] - e_uv[q]) + acc;
        acc = c.ca * u_m.x[q] + acc;
        ru.x[q] = c.cc * u_n.x[q] + acc;
      }
      {   // w
        T acc = BASE ? alpha * bw.x[q] : T(0);
        acc = c.c0 * wc + acc;
        const T sz = w_zp.x[q] + w_zm.x[q];
        acc = cDz * sz + acc;
        acc = cAz * ((w_zp.x[q] - w_zm.x[q]) * (sz + T(2) * wc)) + acc;
        acc = cDx * (wxp + wxm) + acc;
        acc = cAx * (e_uw[q + 1] - e_uw[q]) + acc;
        acc = c.cay * (e_vw_n[q] - e_vw[q]) + acc;
        acc = c.ca * w_m.x[q] + acc;
        rw.x[q] = c.cc * w_n.x[q] + acc;
      }
      {   // v at face j
        T acc = BASE ? alpha * bv.x[q] : T(0);
        acc = c.v0 * vv + acc;
        const T vs = v_n.x[q] + v_m.x[q];
        acc = c.vay * ((v_n.x[q] - v_m.x[q]) * (vs + T(2) * vv)) + acc;
        acc = cDx * (vxp + vxm) + acc;
        acc = cAx * (e_uv[q + 1] - e_uv[q]) + acc;
        acc = cDz * (v_zp.x[q] + v_zm.x[q]) + acc;
        acc = cAz * fz_v[q] + acc;
        acc = c.va * v_m.x[q] + acc;
        rv.x[q] = c.vc * v_n.x[q] + acc;
      }
    }
    if (live) {
      vst<T, V>(a.ou + o, ru);
      vst<T, V>(a.ow + o, rw);
      if (j >= 1) vst<T, V>(a.ov + o, rv);   // interior faces
    }
    // roll
    u_m = u_c; u_c = u_n; u_xp = un_xp;
    w_m = w_c; w_c = w_n;
    v_m = v_c; v_c = v_n; v_xm = vn_xm; v_xp = vn_xp; v_zm = vn_zm;
    if constexpr (!SHARE) wm_zp = w_zp;
#pragma unroll
    for (int q = 0; q < V; ++q) {
      e_uv[q] = e_uv_n[q];
      e_vw[q] = e_vw_n[q];
    }
    e_uv[V] = e_uv_n[V];
  }
  if (live && j1 == ny) vst<T, V>(a.ov + o, BASE ? vldv<T, V>(a.bv + o) : v_c);   // top wall face of v: boundary value
}

template <typename T, int V>
cudaError_t launch_momentum_v(const Geometry& g, const DevTables& tb, const MomArgs<T>& a, const MomCoef& mc,
                              cudaStream_t st, int jlo, int jhi) {
  const int rows = jhi - jlo;
  int tx = 32;                                   // lanes along x: a power of two covering short lines
  while (tx > 1 && (tx / 2) * V >= g.nx) tx /= 2;
  const int tz = MOM_THREADS / tx;
  const int gx = (g.nx + tx * V - 1) / (tx * V), gz = (g.nz + tz - 1) / tz;
  const int jc = momentum_chunk_rows((long long)gx * gz, rows);
  const size_t smem = sizeof(RowCoef<T>) * (size_t)jc;
  const dim3 grid(gx, gz, (rows + jc - 1) / jc), block(tx, tz);
  constexpr bool SH = sizeof(T) == 8;
  const bool base = a.bu != nullptr;
  const void* kern = base ? (const void*)k_momentum<T, V, true, SH> : (const void*)k_momentum<T, V, false, SH>;
  const cudaError_t e = ensure_smem_limit(kern, smem, SH ? sizeof(MVec<T, V>) * 4 * MOM_THREADS : 0);
  if (e != cudaSuccess) return e;
  if (base) k_momentum<T, V, true, SH><<<grid, block, smem, st>>>(g, a, mc, tb.d.inv_dy, tb.d.inv_h, tb.d.a, tb.d.c, jlo, jhi, jc);
  else k_momentum<T, V, false, SH><<<grid, block, smem, st>>>(g, a, mc, tb.d.inv_dy, tb.d.inv_h, tb.d.a, tb.d.c, jlo, jhi, jc);
  return cudaGetLastError();
}

}  // namespace

template <typename T>
cudaError_t launch_momentum(const Geometry& g, const DevTables& tb, const MomArgs<T>& a, cudaStream_t st, int jlo,
                            int jhi) {
  if (jhi < 0) jhi = g.ny;
  if (jlo < 0 || jhi > g.ny || jhi <= jlo) return cudaErrorInvalidValue;
  const double bdtnu = a.bdt * a.nu;
  const MomCoef mc{bdtnu / (g.dx * g.dx), bdtnu / (g.dz * g.dz), -0.25 * a.bdt / g.dx, -0.25 * a.bdt / g.dz,
                   bdtnu, a.bdt * a.fx};
  constexpr int VW = 16 / (int)sizeof(T);
  if constexpr (VW == 2) return launch_momentum_v<T, 2>(g, tb, a, mc, st, jlo, jhi);
  return g.nx % 4 == 0 ? launch_momentum_v<T, VW>(g, tb, a, mc, st, jlo, jhi)
                       : launch_momentum_v<T, 2>(g, tb, a, mc, st, jlo, jhi);
}

template cudaError_t launch_momentum<double>(const Geometry&, const DevTables&, const MomArgs<double>&, cudaStream_t,
                                             int, int);
template cudaError_t launch_momentum<float>(const Geometry&, const DevTables&, const MomArgs<float>&, cudaStream_t,
                                            int, int);

}  // namespace pp
