// Point-source magnification map by the lens polynomial (§4.1: the fifth-
// order polynomial inversion of Eq. 2 solved for a uniform grid of source
// positions, one GPU thread per map pixel), the paper's own map generator.
//
// Per texel centre zeta (FP64 throughout):
//  * The quintic is written in the frame centred on the midpoint of the two
//    masses, w = z - m, lenses at w = -a (primary, eps1) and w = +a
//    (secondary, eps2), a = s/2, omega = zeta - m.  Conjugating Eq. 2 gives
//    conj(w) = N / Dn with Dn = w^2 - a^2 and N = conj(omega) Dn + w + a d,
//    d = eps2 - eps1; substituting back and clearing the denominators
//    (N + a Dn)(N - a Dn) gives
//        (omega - w)(N^2 - a^2 Dn^2) + Dn N + a d Dn^2 = 0,
//    a quintic in w whose roots contain the images.
//  * Its five roots are found together by the Aberth-Ehrlich iteration
//    (each root moves by the Newton step corrected for the other roots),
//    from starting points on a circle enclosing them: in FP32 to a relative
//    move of 1e-5 (FP64 is 1/70 of the FP32 rate on this GPU), then in FP64
//    to 1e-12.
//  * Each root is polished by Newton's method on Eq. 2 itself (the step dw
//    solves f + dw + D conj(dw) = 0, D = d zeta / d conj(z)), which
//    sharpens images next to a low-mass lens where the polynomial's
//    coefficients lose digits.
//  * A root is an image when its Eq. 2 residual, relative to the size of
//    the terms Eq. 2 sums, is below 1e-4 before the polish and below 1e-9
//    after it, and it is not a repeat of an earlier root;
//    A = sum over images of 1/|det J| with det J = 1 - |D|^2 (Eq. 3-4).
//
// That is the general form, 12 000 FP64-pipe instructions per warp of texels
// at some 16 cycles each: 24 ms per 1024^2 map.  k_poly_fast does nearly all
// texels (99.9 % of the maps measured) with a thirtieth of the FP64 work and
// proves its count of images; k_poly_map takes the others.
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include <algorithm>

#include "morse_internal.cuh"

namespace morse {

namespace {

template <typename T>
struct cx {
  T re, im;
};
using cd = cx<double>;
template <typename T>
__device__ __forceinline__ cx<T> mk(T r, T i) { return {r, i}; }
template <typename T>
__device__ __forceinline__ cx<T> add(cx<T> a, cx<T> b) {
  return {a.re + b.re, a.im + b.im};
}
template <typename T>
__device__ __forceinline__ cx<T> sub(cx<T> a, cx<T> b) {
  return {a.re - b.re, a.im - b.im};
}
template <typename T>
__device__ __forceinline__ cx<T> mul(cx<T> a, cx<T> b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename T>
__device__ __forceinline__ cx<T> scl(T s, cx<T> a) {
  return {s * a.re, s * a.im};
}
template <typename T>
__device__ __forceinline__ cx<T> cnj(cx<T> a) { return {a.re, -a.im}; }
template <typename T>
__device__ __forceinline__ T ab2(cx<T> a) {
  return a.re * a.re + a.im * a.im;
}
__device__ __forceinline__ double ab(cd a) { return hypot(a.re, a.im); }
__device__ __forceinline__ float ab(cx<float> a) { return hypotf(a.re, a.im); }
template <typename T>
__device__ __forceinline__ cx<T> dvd(cx<T> a, cx<T> b) {
  // a / b by scaling with the larger component of b (two divisions)
  if (fabs(b.re) >= fabs(b.im)) {
    const T r = b.im / b.re, id = T(1) / (b.re + b.im * r);
    return {(a.re + a.im * r) * id, (a.im - a.re * r) * id};
  }
  const T r = b.re / b.im, id = T(1) / (b.re * r + b.im);
  return {(a.re * r + a.im) * id, (a.im * r - a.re) * id};
}

// Aberth-Ehrlich iterations on the monic quintic with coefficients b
// (z^5 + b4 z^4 + ... + b0) in precision T until the largest relative move
// is below tol or `iters` sweeps are done.
template <typename T>
__device__ __forceinline__ void aberth(const cx<T> (&b)[5], cx<T> (&z)[5],
                                       int iters, T tol) {
  const cx<T> one = mk<T>(1, 0);
  for (int it = 0; it < iters; ++it) {
    T moved = 0;
    for (int t = 0; t < 5; ++t) {
      cx<T> p = one, dp = mk<T>(0, 0);  // p and p' by Horner
      for (int u = 4; u >= 0; --u) {
        dp = add(mul(dp, z[t]), p);
        p = add(mul(p, z[t]), b[u]);
      }
      if (ab2(p) == T(0)) continue;
      const cx<T> nw = dvd(p, dp);  // Newton step p/p'
      cx<T> sum = mk<T>(0, 0);
      for (int u = 0; u < 5; ++u)
        if (u != t) sum = add(sum, dvd(one, sub(z[t], z[u])));
      // Aberth step: nw / (1 - nw * sum)
      const cx<T> step = dvd(nw, sub(one, mul(nw, sum)));
      if (isfinite(step.re) && isfinite(step.im)) {
        z[t] = sub(z[t], step);
        moved = fmax(moved, ab(step) / (T(1) + ab(z[t])));
      }
    }
    if (moved < tol) break;
  }
}

// The roots need only be good starting points for the polish on Eq. 2,
// which takes each image to full precision: FP32 sweeps stop at a relative
// move of 1e-5, FP64 sweeps at 1e-12 (a tighter test would sit at the
// rounding floor of ill-conditioned roots and use up the sweeps).
constexpr int kPolyIters = 30;    // FP64 sweeps at most
constexpr int kPolyItersF = 60;   // FP32 sweeps at most
constexpr int kPolishIters = 8;

// Lens equation in the midpoint frame: omega(w) and D = d omega/d conj(w).
__device__ __forceinline__ void lens(cd w, double a, double e1, double e2,
                                     cd *om, cd *D) {
  const cd wa = mk(w.re + a, -w.im);  // conj(w) + a
  const cd wb = mk(w.re - a, -w.im);  // conj(w) - a
  const cd ia = dvd(mk(1.0, 0.0), wa), ib = dvd(mk(1.0, 0.0), wb);
  *om = sub(sub(w, scl(e1, ia)), scl(e2, ib));
  *D = add(scl(e1, mul(ia, ia)), scl(e2, mul(ib, ib)));
}

// A of texel k by the general form.
__device__ double poly_texel(double s, double q, double L, int npix,
                             size_t k) {
  const double e1 = 1.0 / (1.0 + q), e2 = q / (1.0 + q);
  const double a = 0.5 * s, dl = e2 - e1;
  // midpoint of the masses: the primary sits at -s e2, the secondary at
  // +s e1 (origin at the centre of mass)
  const double m = 0.5 * s * (e1 - e2);
  const double dlt = (2.0 * L) / (double)npix;
  const double a2 = a * a;
  {
    const int i = (int)(k % npix), j = (int)(k / npix);
    const cd om = mk(-L + ((double)i + 0.5) * dlt - m,
                     -L + ((double)j + 0.5) * dlt);
    const cd omc = cnj(om);
    // Dn = w^2 - a^2; N = conj(omega) Dn + w + a d (coefficients by power)
    const cd N0 = mk(-a2 * omc.re + a * dl, -a2 * omc.im);
    const cd N1 = mk(1.0, 0.0);
    const cd N2 = omc;
    // Q = N^2 - a^2 Dn^2, Dn^2 = w^4 - 2 a^2 w^2 + a^4
    cd Q[5];
    Q[0] = sub(mul(N0, N0), mk(a2 * a2 * a2, 0.0));
    Q[1] = scl(2.0, mul(N0, N1));
    Q[2] = add(add(scl(2.0, mul(N0, N2)), mul(N1, N1)),
               mk(2.0 * a2 * a2, 0.0));
    Q[3] = scl(2.0, mul(N1, N2));
    Q[4] = sub(mul(N2, N2), mk(a2, 0.0));
    // p = (omega - w) Q + Dn N + a d Dn^2
    cd c[6];
    for (int t = 0; t < 6; ++t) c[t] = mk(0.0, 0.0);
    for (int t = 0; t < 5; ++t) {
      c[t] = add(c[t], mul(om, Q[t]));
      c[t + 1] = sub(c[t + 1], Q[t]);
    }
    // Dn N = (w^2 - a^2)(N0 + N1 w + N2 w^2)
    c[0] = sub(c[0], scl(a2, N0));
    c[1] = sub(c[1], scl(a2, N1));
    c[2] = add(c[2], sub(N0, scl(a2, N2)));
    c[3] = add(c[3], N1);
    c[4] = add(c[4], N2);
    // a d Dn^2
    const double ad = a * dl;
    c[0] = add(c[0], mk(ad * a2 * a2, 0.0));
    c[2] = add(c[2], mk(-2.0 * ad * a2, 0.0));
    c[4] = add(c[4], mk(ad, 0.0));
    double A_sum = 0.0;
    if (ab2(c[5]) > 0.0) {
      // monic form
      cd b[5];
      for (int t = 0; t < 5; ++t) b[t] = dvd(c[t], c[5]);
      // roots lie within 1 + max |b_t| (Cauchy's bound); start on a circle
      // of half that radius, rotated off the axes
      double R = 0.0;
      for (int t = 0; t < 5; ++t) R = fmax(R, ab(b[t]));
      R = 0.5 * (1.0 + R);
      // roots to single precision in FP32 from a circle of starting
      // points, then to double precision in FP64 (a few cubically
      // converging sweeps)
      cx<float> bf[5], zf[5];
      for (int t = 0; t < 5; ++t) {
        bf[t] = mk((float)b[t].re, (float)b[t].im);
        float sn, cs;
        sincosf(0.4f + 2.0f * (float)CUDART_PI * t / 5.0f, &sn, &cs);
        zf[t] = mk((float)R * cs, (float)R * sn);
      }
      aberth(bf, zf, kPolyItersF, 1e-5f);
      cd z[5];
      bool ok = true;
      for (int t = 0; t < 5; ++t) {
        z[t] = mk((double)zf[t].re, (double)zf[t].im);
        ok = ok && isfinite(z[t].re) && isfinite(z[t].im);
      }
      if (!ok)  // FP32 out of range: start the FP64 sweeps from the circle
        for (int t = 0; t < 5; ++t) {
          double sn, cs;
          sincos(0.4 + 2.0 * CUDART_PI * t / 5.0, &sn, &cs);
          z[t] = mk(R * cs, R * sn);
        }
      aberth(b, z, kPolyIters, 1e-12);
      // polish on Eq. 2 and keep the images
      cd img[5];
      int ni = 0;
      for (int t = 0; t < 5; ++t) {
        cd w = z[t], best = w;
        // the quintic has roots that are not images (3-image sources): they
        // leave Eq. 2 with an O(1) relative residual and are not polished,
        // lest Newton carry them onto an image found already
        {
          cd o, D;
          lens(w, a, e1, e2, &o, &D);
          const double sc0 = ab(w) + ab(om) + e1 / ab(mk(w.re + a, w.im)) +
                             e2 / ab(mk(w.re - a, w.im));
          if (!(ab(sub(o, om)) < 1e-4 * sc0)) continue;
        }
        double best_r = CUDART_INF;
        for (int it = 0; it <= kPolishIters; ++it) {
          cd o, D;
          lens(w, a, e1, e2, &o, &D);
          const cd f = sub(o, om);
          const double r = ab(f);
          if (!(r < best_r)) break;  // no longer improving: at the floor
          best_r = r;
          best = w;
          if (r == 0.0 || it == kPolishIters) break;
          const double det = 1.0 - ab2(D);
          if (det == 0.0) break;
          const cd dw = scl(1.0 / det, sub(mul(D, cnj(f)), f));
          w = add(w, dw);
          if (ab2(dw) <= 1e-32 * (1.0 + ab2(w))) {  // converged: one check
            lens(w, a, e1, e2, &o, &D);
            const double r2 = ab(sub(o, om));
            if (r2 < best_r) {
              best_r = r2;
              best = w;
            }
            break;
          }
        }
        // residual relative to the size of the terms of Eq. 2
        const double sc = ab(best) + ab(om) +
                          e1 / ab(mk(best.re + a, best.im)) +
                          e2 / ab(mk(best.re - a, best.im));
        if (!(best_r < 1e-9 * sc)) continue;
        bool dup = false;
        for (int u = 0; u < ni; ++u)
          if (ab(sub(best, img[u])) <= 1e-9 * (1.0 + ab(img[u]))) dup = true;
        if (dup) continue;
        img[ni++] = best;
        cd o, D;
        lens(best, a, e1, e2, &o, &D);
        A_sum += 1.0 / fabs(1.0 - ab2(D));
      }
    }
    return A_sum;
  }
}

// The general form of every texel, or (LEFT) of those the fast form left, NaN:
// a block collects them from a tile of texels in shared memory first, so that
// its warps are full.
//
// A texel takes a warp half a millisecond or more whether its other lanes
// have one too, so what counts is that the texels spread over the SMs: a
// thread takes one at a time, and the tiles of a small map are small
// (launch_poly_map).  Every map in tiles of 16 texels per thread took 35 ms
// at 64^2 and 31 at 256^2, so 2.4 and 6.8 (q = 1e-9).
constexpr int kPolyThreads = 128, kPolyTile = 16 * kPolyThreads;

template <bool LEFT>
__global__ void __launch_bounds__(kPolyThreads)
    k_poly_map(double s, double q, double L, int npix, int tile,
               float *__restrict__ A) {
  const size_t n = (size_t)npix * npix;
  if (!LEFT) {
    for (size_t k = blockIdx.x * (size_t)kPolyThreads + threadIdx.x; k < n;
         k += gridDim.x * (size_t)kPolyThreads)
      A[k] = __double2float_rn(poly_texel(s, q, L, npix, k));
    return;
  }
  __shared__ unsigned s_q[kPolyTile], s_n;
  for (size_t c0 = blockIdx.x * (size_t)tile; c0 < n;
       c0 += gridDim.x * (size_t)tile) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < tile; t += kPolyThreads)
      if (c0 + t < n && isnan(A[c0 + t]))
        s_q[atomicAdd(&s_n, 1u)] = (unsigned)t;
    __syncthreads();
    const unsigned m = s_n;
    for (unsigned t = threadIdx.x; t < m; t += kPolyThreads) {
      const size_t k = c0 + s_q[t];
      A[k] = __double2float_rn(poly_texel(s, q, L, npix, k));
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------ fast form
// Origin at the lighter lens B (mass mb), the other (ma) at h on the axis:
//     omega = w - ma/(conj(w) - h) - mb/conj(w).
// With N = conj(omega) w^2 + (1 - conj(omega) h) w - mb h and A = N - h P,
// P = w (w - h), conj(w) = N/P and
//     (w - omega) A N - P (ma N + mb A) = 0.
// About the lighter lens its cluster of roots (of size sqrt(mb)) is held by
// the low coefficients to their own relative precision, so FP32 resolves it:
// coefficients in FP64, rounded, and Aberth-Ehrlich in FP32 from radii of
// the Newton polygon of |b_t| (Bini 1996), which takes 5 to 6 sweeps where a
// circle of Cauchy's bound takes some 20.
//
// A root whose FP32 residual of Eq. 2 is below 0.2 % of its terms is a
// candidate, polished by Newton on Eq. 2 (twice in FP32, then in FP64 until
// the step changes 1/|det J| by less than 1e-12 of it, or for the first time
// by less than 2e-9, which near a caustic is all that FP64 allows, and one
// step more: 7 of 4.2e7 texels differ from the general form's by an FP32 ulp;
// without that step 749).  The texel is kept only if
// every candidate became an image of its own or is shown to be none
// (spurious), they are 3 or 5, and their parities add up to -1 (one more
// saddle than minima and maxima, for two point lenses).  Two point lenses
// have 3 or 5 images, so five are all, and three are all once a single root
// of the quintic is known to be no image: a spurious candidate, or one of the
// other roots, by a bound that needs no converged root (no_image) or else
// polished in FP64 (spurious).  (Without that proof, a root that the sweeps
// had not brought to its place passed for no image: 51 of 1e8 texels about
// the caustics of lenses of s = 2.5 to 28 lost a pair of images.)
// Emulated on the CPU: of 1e8 texels about the caustics of lenses of s = 2.5 to
// 28, and 1.8e7 over s 0.01 to 30, q 1e-8 to 10, L 0.02 to 100, none kept
// differs from the general form's value by 1e-5, and fewer than 1 in 1000 is
// left to that form where s is 0.3 to 3 (0.5 % of close lenses' maps, 17 %
// over the whole range).  1024^2 map: 23.9 -> 1.12 ms.
using cf = cx<float>;

__device__ __forceinline__ float rcpf(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ cf divf(cf a, cf b) {
  const float r = rcpf(ab2(b));
  return {(a.re * b.re + a.im * b.im) * r, (a.im * b.re - a.re * b.im) * r};
}
// 1/x by two Newton steps from the FP32 reciprocal (relative error a few
// 2^-53; x outside FP32's range gives infinity or NaN)
__device__ __forceinline__ double rcpd(double x) {
  double r = (double)rcpf((float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// coefficients of the quintic, c[5] the leading one
__device__ __forceinline__ void quintic(double mb, double h, cd om,
                                        cd (&c)[6]) {
  const cd oc = cnj(om);
  const double n0 = -mb * h, hh = h * h;
  const cd n1 = mk(1.0 - oc.re * h, -oc.im * h);
  const cd a1 = mk(n1.re + hh, n1.im), a2 = mk(oc.re - h, oc.im);
  const cd s1 = add(a1, n1), s2 = add(a2, oc);
  const double k0 = n0 * n0;
  const cd k1 = scl(n0, s1);
  const cd k2 = add(scl(n0, s2), mul(a1, n1));
  const cd k3 = add(mul(a2, n1), mul(a1, oc));
  const cd k4 = mul(a2, oc);
  const cd m2 = mk(oc.re - mb * h, oc.im);
  const cd m1 = mk(n1.re + mb * hh, n1.im);
  c[0] = scl(-k0, om);
  c[1] = mk(k0 + h * n0, 0.0);
  c[1] = sub(c[1], mul(om, k1));
  c[2] = sub(sub(k1, mul(om, k2)), mk(n0 - h * m1.re, -h * m1.im));
  c[3] = sub(sub(k2, mul(om, k3)), sub(m1, scl(h, m2)));
  c[4] = sub(sub(k3, mul(om, k4)), m2);
  c[5] = k4;
}

// Whether the root of the quintic near z is no image for certain: polished
// in FP64 as a root of the quintic, it leaves Eq. 2 by more than 1e-6 of its
// terms.  (Near a caustic's outside the two roots about to become images
// are candidates too: a few texels per map, whose general form would keep
// one warp busy for half a millisecond.)
__device__ __noinline__ bool spurious(double mb, double ma, double h, cd om,
                                      cf z) {
  cd c[6];
  quintic(mb, h, om, c);
  cd w = mk((double)z.re, (double)z.im);
  bool done = false;
  for (int it = 0; it < 8 && !done; ++it) {
    cd p = c[5], dp = mk(0.0, 0.0);
    for (int u = 4; u >= 0; --u) {
      dp = add(mul(dp, w), p);
      p = add(mul(p, w), c[u]);
    }
    const double r = 1.0 / ab2(dp);
    const cd st = mk((p.re * dp.re + p.im * dp.im) * r,
                     (p.im * dp.re - p.re * dp.im) * r);
    w = sub(w, st);
    done = ab2(st) < 1e-22 * ab2(w);
  }
  if (!done) return false;
  const double xa = w.re - h;
  const double ra = 1.0 / (xa * xa + w.im * w.im), rb = 1.0 / ab2(w);
  const double fr = w.re - ma * xa * ra - mb * w.re * rb - om.re;
  const double fi = w.im - ma * w.im * ra - mb * w.im * rb - om.im;
  const double sc = sqrt(ab2(w)) + sqrt(ab2(om)) + ma * sqrt(ra) +
                    mb * sqrt(rb);
  return fr * fr + fi * fi > 1e-12 * sc * sc;
}

// Whether a disc about z holds a root of the monic quintic b and no image, by
// FP32 arithmetic alone: z may be far from converged.  f: |residual of Eq. 2|
// at z, ra and rb: 1/|z - h|^2 and 1/|z|^2.
//  * 5 |p/p'| about any point is the radius of a disc with a root.  Horner's
//    rounding and that of the coefficients are below 40 u sum |b_t| |z|^t.
//  * Within rho of z the residual changes by less than
//    rho (1 + 2 ma / |z - h|^2 + 2 mb / |z|^2) when 2 rho is below both
//    distances.  f's own rounding is some 1e-5 of its terms, f above 0.2 %.
__device__ __forceinline__ bool no_image(const cf (&b)[5], cf z, float f,
                                         float ra, float rb, float ma,
                                         float mb) {
  cf p = mk(1.f, 0.f), dp = mk(0.f, 0.f);
  float s = 1.f, ds = 0.f;  // the same of the absolute values, or above
  const float az = sqrt_approx(ab2(z));
#pragma unroll
  for (int u = 4; u >= 0; --u) {
    dp = add(mul(dp, z), p);
    p = add(mul(p, z), b[u]);
    ds = ds * az + s;
    s = s * az + (fabsf(b[u].re) + fabsf(b[u].im));
  }
  const float e = 40.f / 16777216.f;
  const float num = 5.f * (sqrt_approx(ab2(p)) + e * s);  // rho = num / den
  const float den = sqrt_approx(ab2(dp)) - e * ds;
  return den > 0.f && 4.f * num * num * fmaxf(ra, rb) < den * den &&
         2.f * num * (1.f + 2.f * (ma * ra + mb * rb)) < f * den;
}

__global__ void __launch_bounds__(kPolyThreads)
    k_poly_fast(double mb, double ma, double xb, double h, double L, int npix,
                float *__restrict__ A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npix) return;
  const int j = blockIdx.y;
  const double dlt = (2.0 * L) / (double)npix;
  const cd om = mk(-L + ((double)i + 0.5) * dlt - xb,
                   -L + ((double)j + 0.5) * dlt);
  cf b[5];
  {
    cd c[6];
    quintic(mb, h, om, c);
    const cf lead = mk((float)c[5].re, (float)c[5].im);
#pragma unroll
    for (int t = 0; t < 5; ++t)
      b[t] = divf(mk((float)c[t].re, (float)c[t].im), lead);
  }
  cf z[5];
  {
    // radii: the slopes of the upper hull of (t, log2 |b_t|), b_5 = 1
    float lb[6];
#pragma unroll
    for (int t = 0; t < 5; ++t)
      lb[t] = 0.5f * __log2f(fmaxf(ab2(b[t]), 1e-37f));
    lb[5] = 0.f;
    const float cs[5] = {0.92106099f, -0.08573640f, -0.97404902f,
                         -0.51625902f, 0.65498345f};
    const float sn[5] = {0.38941834f, 0.99631784f, 0.22633998f,
                         -0.85643203f, -0.75564413f};
#pragma unroll
    for (int t = 0; t < 5; ++t) {
      float lo = 3e38f;
#pragma unroll
      for (int u = 0; u <= t; ++u) {
        float hi = -3e38f;
#pragma unroll
        for (int v = t + 1; v < 6; ++v)
          hi = fmaxf(hi, (lb[v] - lb[u]) * (1.f / (float)(v - u)));
        lo = fminf(lo, hi);
      }
      const float r = exp2f(-lo);
      z[t] = mk(r * cs[t], r * sn[t]);
    }
  }
  for (int it = 0; it < 24; ++it) {
    bool moved = false;
#pragma unroll
    for (int t = 0; t < 5; ++t) {
      cf p = mk(1.f, 0.f), dp = mk(0.f, 0.f);
#pragma unroll
      for (int u = 4; u >= 0; --u) {
        dp = add(mul(dp, z[t]), p);
        p = add(mul(p, z[t]), b[u]);
      }
      cf sum = mk(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 5; ++u)
        if (u != t) {
          const cf d = sub(z[t], z[u]);
          const float r = rcpf(ab2(d));
          sum = add(sum, mk(d.re * r, -d.im * r));
        }
      const cf nw = divf(p, dp);
      const cf st = divf(nw, sub(mk(1.f, 0.f), mul(nw, sum)));
      if (isfinite(st.re) && isfinite(st.im)) {
        z[t] = sub(z[t], st);
        moved |= ab2(st) > 9e-10f * ab2(z[t]);
      }
    }
    if (!moved) break;
  }
  // candidates, to the front
  const float hf = (float)h, maf = (float)ma, mbf = (float)mb;
  const cf omf = mk((float)om.re, (float)om.im);
  cf w0[5], z0[5];  // their polished and their own places
  int ni = 0;
  cf zn = mk(0.f, 0.f);  // the other root that leaves Eq. 2 the furthest
  float fn = 0.f, sc_n = 1.f, ra_n = 0.f, rb_n = 0.f;
#pragma unroll
  for (int t = 0; t < 5; ++t) w0[t] = z0[t] = mk(0.f, 0.f);
#pragma unroll
  for (int t = 0; t < 5; ++t) {
    cf w = z[t];
    bool cand = false;
#pragma unroll
    for (int it = 0; it < 3; ++it) {  // the residual, then two Newton steps
      const float xa = w.re - hf;
      const float ra = rcpf(xa * xa + w.im * w.im), rb = rcpf(ab2(w));
      const cf ia = mk(xa * ra, w.im * ra), ib = mk(w.re * rb, w.im * rb);
      const cf f = mk(w.re - maf * ia.re - mbf * ib.re - omf.re,
                      w.im - maf * ia.im - mbf * ib.im - omf.im);
      if (it == 0) {
        const float sc = sqrtf(ab2(w)) + sqrtf(ab2(omf)) +
                         maf * sqrtf(ra) + mbf * sqrtf(rb);
        // (a NaN is a candidate, which will not converge)
        const float af = sqrtf(ab2(f));
        cand = !(af >= 0.002f * sc);
        if (!cand && af * sc_n > fn * sc) {
          zn = w;
          fn = af;
          sc_n = sc;
          ra_n = ra;
          rb_n = rb;
        }
      }
      const cf D = add(scl(maf, mul(ia, ia)), scl(mbf, mul(ib, ib)));
      const float rd = rcpf(1.f - ab2(D));
      const cf dw = scl(rd, sub(mul(D, cnj(f)), f));
      if (it > 0 && ab2(dw) < 1e-4f * ab2(w)) w = add(w, dw);
    }
    if (cand) {
#pragma unroll
      for (int u = 0; u < 5; ++u)
        if (u == ni) {
          w0[u] = w;
          z0[u] = z[t];
        }
      ++ni;
    }
  }
  // three images are all there are when one root is known not to be one: a
  // candidate shown spurious, or another root (here, before the FP64 steps:
  // after them the coefficients' registers cost a block per SM)
  const bool three = ni == 3 && no_image(b, zn, fn, ra_n, rb_n, maf, mbf);
  double A_sum = 0.0;
  int parity = 0, images = 0;
  bool ok = ni >= 3;
#pragma unroll
  for (int t = 0; t < 5; ++t) {
    if (t >= ni || !ok) break;
    double x = (double)w0[t].re, y = (double)w0[t].im;
    bool done = false, near = false;
    for (int it = 0; it < 7 && !done; ++it) {
      const double xa = x - h, yy = y * y;
      const double ra = rcpd(fma(xa, xa, yy)), rb = rcpd(fma(x, x, yy));
      const double iar = xa * ra, iai = y * ra, ibr = x * rb, ibi = y * rb;
      const double fr = fma(-mb, ibr, fma(-ma, iar, x - om.re));
      const double fi = fma(-mb, ibi, fma(-ma, iai, y - om.im));
      const double Dr = fma(ma, fma(iar, iar, -iai * iai),
                            mb * fma(ibr, ibr, -ibi * ibi));
      const double Di = 2.0 * fma(ma, iar * iai, mb * (ibr * ibi));
      const double det = 1.0 - fma(Dr, Dr, Di * Di);
      const double rd = rcpd(det);
      const double dx = (fma(Dr, fr, Di * fi) - fr) * rd;
      const double dy = (fma(Di, fr, -Dr * fi) - fi) * rd;
      // |d (1/det)| <= |d|D|^2/dw| |dw| / det^2, d|D|^2/dw <= 2 |D| |D'|
      const float ga = sqrtf((float)ra), gb = sqrtf((float)rb);
      const float g = 4.f * sqrtf((float)(Dr * Dr + Di * Di)) *
                      (maf * ga * ga * ga + mbf * gb * gb * gb);
      const float st = sqrtf((float)dx * (float)dx + (float)dy * (float)dy);
      const float re = sqrtf((float)fr * (float)fr + (float)fi * (float)fi);
      const float sc = sqrtf((float)(x * x) + (float)yy) + sqrtf(ab2(omf)) +
                       maf * ga + mbf * gb;
      // one step more within the bound, unless it would not show
      const float mv = g * st, ad = fabsf((float)det);
      const bool in = mv <= 2e-9f * ad && re < 1e-9f * sc;
      if (in && (near || mv <= 1e-12f * ad)) {
        done = true;
        w0[t] = mk((float)x, (float)y);
#pragma unroll
        for (int u = 0; u < t; ++u)  // (w0 of no image: NaN)
          if (ab2(sub(w0[t], w0[u])) < 1e-12f * (1e-6f + ab2(w0[t])))
            done = false;
        if (!done) break;
        ++images;
        A_sum += fabs(rd);
        parity += det > 0.0 ? 1 : -1;
      } else {
        near |= in;
        x += dx;
        y += dy;
      }
    }
    if (!done) {
      w0[t] = mk(CUDART_NAN_F, CUDART_NAN_F);
      ok = spurious(mb, ma, h, om, z0[t]);
    }
  }
  if (images == 3 && ni == 3 && !three)
    ok = ok && spurious(mb, ma, h, om, zn);
  A[(size_t)j * npix + i] =
      ok && (images == 3 || images == 5) && parity == -1
          ? __double2float_rn(A_sum)
          : CUDART_NAN_F;
}

}  // namespace

cudaError_t launch_poly_map(double s, double q, double L, int npix, float *A,
                            int sm_count, cudaStream_t st) {
  // the fast form where FP32 holds the lens and the map: its checks leave a
  // texel it cannot settle to the general form in any case (beyond s = 30 that
  // would be most of them: FP32 Aberth does not converge there)
  const double e1 = 1.0 / (1.0 + q), e2 = q / (1.0 + q);
  const bool second = e2 <= e1;  // the lighter lens
  const double mb = second ? e2 : e1, ma = second ? e1 : e2;
  const double x1 = -s * e2, x2 = s * e1;
  const double xb = second ? x2 : x1, h = second ? x1 - x2 : x2 - x1;
  const bool fast = mb >= 1e-8 && s >= 1e-2 && s <= 30.0 && L <= 100.0;
  if (fast) {
    const dim3 grid((unsigned)((npix + kPolyThreads - 1) / kPolyThreads),
                    (unsigned)npix);
    k_poly_fast<<<grid, kPolyThreads, 0, st>>>(mb, ma, xb, h, L, npix, A);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // one texel per thread; or tiles two to an SM, of one to 16 texels per
  // thread (larger ones only where there are tiles enough: fuller warps)
  const size_t n = (size_t)npix * npix;
  size_t tile = kPolyThreads;
  if (fast) {
    tile = (n / (2 * (size_t)sm_count) + kPolyThreads) / kPolyThreads *
           kPolyThreads;
    tile = std::min<size_t>(tile, kPolyTile);
  }
  const size_t blocks =
      std::min((n + tile - 1) / tile, (size_t)sm_count * 16);
  if (fast)
    k_poly_map<true><<<(unsigned)blocks, kPolyThreads, 0, st>>>(
        s, q, L, npix, (int)tile, A);
  else
    k_poly_map<false><<<(unsigned)blocks, kPolyThreads, 0, st>>>(
        s, q, L, npix, (int)tile, A);
  return cudaGetLastError();
}

}  // namespace morse
