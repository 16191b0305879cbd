// Stockham stages whose twiddles are fused into the butterflies (FP64 transforms, whose bound is
// the FP64 issue rate of two instructions per clock and SM).
//
// A twiddled radix-2 butterfly a +- w b with w = c (1 + i t), c = cos, t = tan of the twiddle's
// angle, is 2 FMAs for b' = (1 + i t) b and 4 for a +- c b' (Linzer and Feig, 1993), instead of 4
// for the product w b and 4 additions.  A radix-8 stage is three levels of four such butterflies,
// with the stage's twiddles pushed down the levels (angles 4k, 2k, k and k + L/8): 72 instructions
// against 92, with 4 table entries against 7.  |c t| <= 1 bounds the error of b' c by that of the
// plain product, at any angle (at a quarter turn c is 6e-17 and t its inverse).
// Per point a 512-point transform (8 x 8 x 8) takes 24.5 instructions instead of 31.  At 512x384x512
// the FP64 passes went from 4.69 / 2.63 / 3.39 ms (divergence and x, z, inverse x) to 3.56 / 2.18 /
// 2.52 ms.  The transform itself is the more accurate one: of random data (this code compiled for the
// host, 40 lines a length) its rms error against an extended-precision DFT is 0.90 to 1.03 (mean 0.96)
// times that of the plain butterflies with the same unit roots at 18 lengths from 16 to 1024 (512
// points: 1.87e-16 and 2.01e-16; 108, the worst: 1.97e-16 and 1.93e-16).  A whole call's distance from another FP64 computation does not resolve that (two steps
// at 512x384x512: 8.0e-15 to 9.6e-15 between seeds and runs, 9.0e-15 with the plain ones).
#pragma once

#include "fft_static.cuh"

namespace pp {

// One table entry: (cos, tan) of 2 pi n / L, as cplx<T>.
// (o0, o1) = a +- w b, w = e^{SIGN i theta}; Q: w times the quarter turn SIGN i.
template <typename T, int SIGN, bool Q>
__device__ __forceinline__ void lf_bfly(cplx<T> a, cplx<T> b, cplx<T> w, cplx<T>& o0, cplx<T>& o1) {
  const T t = SIGN < 0 ? -w.y : w.y, c = w.x;
  const T bx = fma(-t, b.y, b.x), by = fma(t, b.x, b.y);
  if constexpr (!Q) {
    o0 = mk<T>(fma(c, bx, a.x), fma(c, by, a.y));
    o1 = mk<T>(fma(-c, bx, a.x), fma(-c, by, a.y));
  } else {
    const cplx<T> p = mk<T>(fma(-c, by, a.x), fma(c, bx, a.y)), m = mk<T>(fma(c, by, a.x), fma(-c, bx, a.y));
    o0 = SIGN > 0 ? p : m;
    o1 = SIGN > 0 ? m : p;
  }
}

// a +- r u, with the factor in the FMAs.
template <typename T>
__device__ __forceinline__ void fma_pair(cplx<T> a, cplx<T> u, T r, cplx<T>& o0, cplx<T>& o1) {
  o0 = mk<T>(fma(r, u.x, a.x), fma(r, u.y, a.y));
  o1 = mk<T>(fma(-r, u.x, a.x), fma(-r, u.y, a.y));
}

// R-point DFT without twiddles, the constant factors folded into FMAs.
template <typename T, int R, int SIGN>
__device__ __forceinline__ void lf_dft(cplx<T>* v) {
  if constexpr (R == 8) {
    const T r = T(0.70710678118654752440084436210485);
    cplx<T> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft4<T, SIGN>(e);
    dft4<T, SIGN>(o);
    // e^{SIGN i pi/4} o1 = r u1, e^{SIGN 3 i pi/4} o3 = r u3
    const cplx<T> u1 = SIGN < 0 ? mk<T>(o[1].x + o[1].y, o[1].y - o[1].x) : mk<T>(o[1].x - o[1].y, o[1].y + o[1].x);
    const cplx<T> w3 = SIGN < 0 ? mk<T>(o[3].x + o[3].y, o[3].y - o[3].x) : mk<T>(o[3].x - o[3].y, o[3].y + o[3].x);
    const cplx<T> u3 = mul_i(w3, SIGN), o2 = mul_i(o[2], SIGN);
    v[0] = e[0] + o[0];
    v[4] = e[0] - o[0];
    fma_pair(e[1], u1, r, v[1], v[5]);
    v[2] = e[2] + o2;
    v[6] = e[2] - o2;
    fma_pair(e[3], u3, r, v[3], v[7]);
  } else if constexpr (R == 3) {
    const T h = T(0.86602540378443864676372317075294);
    const cplx<T> s = v[1] + v[2], d = mul_i(v[1] - v[2], SIGN);
    const cplx<T> m = mk<T>(fma(T(-0.5), s.x, v[0].x), fma(T(-0.5), s.y, v[0].y));
    v[0] = v[0] + s;
    fma_pair(m, d, h, v[1], v[2]);
  } else {
    dft_r<T, R, SIGN>(v);
  }
}

// R-point DFT of v[r] w^r with w = e^{SIGN 2 pi i n / L}; tw: the table of L entries, n (R - 1) < L.
template <typename T, int R, int SIGN, int L>
__device__ __forceinline__ void lf_dft_tw(cplx<T>* v, const cplx<T>* __restrict__ tw, int n) {
  if constexpr (R == 8) {
    const cplx<T> w1 = ldg_c(tw + n), w2 = ldg_c(tw + 2 * n), w4 = ldg_c(tw + 4 * n), w18 = ldg_c(tw + n + L / 8);
    cplx<T> p[4], m[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) lf_bfly<T, SIGN, false>(v[r], v[r + 4], w4, p[r], m[r]);
    cplx<T> pp[2], pm[2], mp[2], mm[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      lf_bfly<T, SIGN, false>(p[r], p[r + 2], w2, pp[r], pm[r]);
      lf_bfly<T, SIGN, true>(m[r], m[r + 2], w2, mp[r], mm[r]);
    }
    lf_bfly<T, SIGN, false>(pp[0], pp[1], w1, v[0], v[4]);
    lf_bfly<T, SIGN, true>(pm[0], pm[1], w1, v[2], v[6]);
    lf_bfly<T, SIGN, false>(mp[0], mp[1], w18, v[1], v[5]);
    lf_bfly<T, SIGN, true>(mm[0], mm[1], w18, v[3], v[7]);
  } else if constexpr (R == 4) {
    const cplx<T> w1 = ldg_c(tw + n), w2 = ldg_c(tw + 2 * n);
    cplx<T> p[2], m[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) lf_bfly<T, SIGN, false>(v[r], v[r + 2], w2, p[r], m[r]);
    lf_bfly<T, SIGN, false>(p[0], p[1], w1, v[0], v[2]);
    lf_bfly<T, SIGN, true>(m[0], m[1], w1, v[1], v[3]);
  } else if constexpr (R == 2) {
    const cplx<T> a = v[0], b = v[1];
    lf_bfly<T, SIGN, false>(a, b, ldg_c(tw + n), v[0], v[1]);
  } else {
    static_assert(R == 3, "radices 8, 4, 3, 2");
    const T h = T(0.86602540378443864676372317075294);
    const cplx<T> w1 = ldg_c(tw + n), w2 = ldg_c(tw + 2 * n);
    const T t1 = SIGN < 0 ? -w1.y : w1.y;
    const cplx<T> b = mk<T>(w1.x * fma(-t1, v[1].y, v[1].x), w1.x * fma(t1, v[1].x, v[1].y));
    cplx<T> s, d;
    lf_bfly<T, SIGN, false>(b, v[2], w2, s, d);
    d = mul_i(d, SIGN);
    const cplx<T> m = mk<T>(fma(T(-0.5), s.x, v[0].x), fma(T(-0.5), s.y, v[0].y));
    v[0] = v[0] + s;
    fma_pair(m, d, h, v[1], v[2]);
  }
}

// One in-place stage (the data movement of stage_inplace).
template <typename T, int L, int S, int SIGN, int B, int THREADS, int ES, int BS, bool MAPB, int MAXR>
__device__ __forceinline__ void stage_lf(cplx<T>* buf, const cplx<T>* __restrict__ tw) {
  constexpr Radix F = factorize(L, MAXR);
  constexpr int R = F.r[S];
  constexpr int Ns = span_before(L, S, MAXR);
  constexpr int NBF = L / R;
  constexpr int TOTAL = NBF * B;
  constexpr int PER = (TOTAL + THREADS - 1) / THREADS;
  constexpr int TSTRIDE = L / (Ns * R);
  cplx<T> v[PER][R];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int idx = threadIdx.x + q * THREADS;
    const int t = MAPB ? idx % B : idx / NBF, j = MAPB ? idx / B : idx % NBF;
    if (TOTAL % THREADS == 0 || idx < TOTAL) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[q][r] = buf[padi<T>(t * BS + (j + r * NBF) * ES)];
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int idx = threadIdx.x + q * THREADS;
    const int t = MAPB ? idx % B : idx / NBF, j = MAPB ? idx / B : idx % NBF;
    if (TOTAL % THREADS == 0 || idx < TOTAL) {
      const int k = j % Ns;
      if constexpr (Ns > 1) lf_dft_tw<T, R, SIGN, L>(v[q], tw, k * TSTRIDE);
      else lf_dft<T, R, SIGN>(v[q]);
      const int base = (j - k) * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) buf[padi<T>(t * BS + (base + r * Ns) * ES)] = v[q][r];
    }
  }
  __syncthreads();
}

template <typename T, int L, int S, int SIGN, int B, int THREADS, int ES, int BS, bool MAPB, int MAXR>
__device__ __forceinline__ void stages_lf(cplx<T>* buf, const cplx<T>* __restrict__ tw) {
  constexpr Radix F = factorize(L, MAXR);
  if constexpr (S < F.n) {
    stage_lf<T, L, S, SIGN, B, THREADS, ES, BS, MAPB, MAXR>(buf, tw);
    stages_lf<T, L, S + 1, SIGN, B, THREADS, ES, BS, MAPB, MAXR>(buf, tw);
  }
}

// fft_static with the fused butterflies; tw: the (cos, tan) table of L entries.
template <typename T, int L, int SIGN, int B, int THREADS, int ES, int BS, bool MAPB>
__device__ __forceinline__ void fft_lf(cplx<T>* buf, const cplx<T>* __restrict__ tw) {
  static_assert(factorizable(L), "FFT length must be 2^a 3^b");
  stages_lf<T, L, 0, SIGN, B, THREADS, ES, BS, MAPB, 8>(buf, tw);
}

// The even/odd split of a real line's half-length transform for the bins k and M - k at once
// (0 < k < M/2): with s = Z_k + conj Z_{M-k}, d = Z_k - conj Z_{M-k} and W = e^{-2 pi i k/Nx},
// 2 X_k = s - i W d and 2 X_{M-k} = conj(s + i W d); the product takes the fused form (w: the
// (cos, tan) of 2 pi k / Nx).  10 instructions for both bins, where each took 12; the factor 1/2 is
// in the input.
template <typename T>
__device__ __forceinline__ void fwd_post_pair(cplx<T> Zk, cplx<T> Zm, cplx<T> w, cplx<T>& Xk, cplx<T>& Xm) {
  const cplx<T> s = mk<T>(Zk.x + Zm.x, Zk.y - Zm.y), d = mk<T>(Zk.x - Zm.x, Zk.y + Zm.y);
  const T dx = fma(w.y, d.y, d.x), dy = fma(-w.y, d.x, d.y);
  Xk = mk<T>(fma(w.x, dy, s.x), fma(-w.x, dx, s.y));
  Xm = mk<T>(fma(-w.x, dy, s.x), fma(-w.x, dx, -s.y));
}

// Its inverse (inv_pre for k and M - k at once): Z_k = s + i conj(W) d, Z_{M-k} = conj(s - i conj(W) d)
// with s = X_k + conj X_{M-k}, d = X_k - conj X_{M-k}.
template <typename T>
__device__ __forceinline__ void inv_pre_pair(cplx<T> Xk, cplx<T> Xm, cplx<T> w, cplx<T>& Zk, cplx<T>& Zm) {
  const cplx<T> s = mk<T>(Xk.x + Xm.x, Xk.y - Xm.y), d = mk<T>(Xk.x - Xm.x, Xk.y + Xm.y);
  const T dx = fma(-w.y, d.y, d.x), dy = fma(w.y, d.x, d.y);
  Zk = mk<T>(fma(-w.x, dy, s.x), fma(w.x, dx, s.y));
  Zm = mk<T>(fma(w.x, dy, s.x), fma(w.x, dx, -s.y));
}

}  // namespace pp
