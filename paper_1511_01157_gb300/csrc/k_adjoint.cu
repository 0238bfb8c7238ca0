// Adjoint gradient of the profiled chi^2 and the batched Levenberg-Marquardt
// refinement of grid minima.
//
// The paper refines its coarse-grid seeds (§4.4) by MCMC with finite-source
// magnifications (§5).  This library refines them on the same point-source
// map instead: chi^2(theta), theta = (t0, tE, u0, alpha), with (Fs, Fb)
// profiled out by the 2x2 solve of Eq. 6.  Because (Fs, Fb) minimise chi^2
// for every theta, the envelope theorem gives
//     d chi^2 / d theta_k = sum_i -2 w_i r_i Fs dA_i/dtheta_k,
// r_i = F_i - Fs A_i - Fb, and the Gauss-Newton matrix
//     H_kl = sum_i w_i Fs^2 (dA_i/dtheta_k)(dA_i/dtheta_l).
// dA/dtheta follows the lookup: inside the map the bilinear gradient in
// pixel units times dy/dtheta / Delta; outside, the single-lens dA/du times
// du/dtheta.  With tau = (t - t0)/tE, y = tau (c, s) + u0 (-s, c),
// (c, s) = (cos alpha, sin alpha), G = grad_y A, Gp = G.(c, s) and
// Gn = G.(-s, c):
//     dA/dt0 = -Gp / tE,   dA/dtE = -tau Gp / tE,
//     dA/du0 = Gn,         dA/dalpha = tau Gn - u0 Gp.
// One warp per trajectory; FP32 per lane, FP64 across lanes.
// Inside-map epoch loops unrolled: the sweeps wait on texel gathers from L2,
// and four or eight independent gathers per lane are in flight.
#include <algorithm>

#include <cuda_runtime.h>
#include <math_constants.h>

#include "morse_internal.cuh"
#include "search_common.cuh"

namespace morse {

namespace {

using namespace dev;

// GB300 design.  A block of kAdjWarps warps takes kAdjWarps trajectories,
// one warp each for the two epoch sweeps (lanes over epochs, as the search).
// The per-trajectory FP64 work -- sin/cos of alpha, the track constants and
// epoch ranges, the 2x2 solve, and the final assembly of the gradient and
// the Gauss-Newton matrix -- is done by warp 0 with one lane per
// trajectory: GB300's FP64 rate is 1/73 of its FP32 rate, and a warp-wide
// FP64 instruction costs the same whether one lane or 32 need it.  The
// light curve is staged in shared memory when it fits.
//
// Sweep 1 is the search's phase 1 (same device function, same sums), so
// Fs, Fb and chi^2 at a grid point equal the search's to the last bit.
// Sweep 2 takes the residuals r = F - Fs A - Fb (chi^2 summed as the
// search's phase 2 sums it) and accumulates the gradient in the map's
// pixel axes: with g = (gx, gy) = Delta grad_y A (the bilinear cell's
// slopes inside the map, Delta D y with D = (dA/du)/u outside),
// X1 = sum w r gx, Y1 = sum w r gy, X2 = sum w r tau gx, Y2 = sum w r tau gy.
// Rotated once per trajectory into the track's axes, Gp = g.(c, s)/Delta
// and Gn = g.(-s, c)/Delta, they give every component of
//     d chi^2/d theta = -2 Fs sum w r dA/dtheta,
//     dA/dt0 = -Gp/tE, dA/dtE = -tau Gp/tE, dA/du0 = Gn,
//     dA/dalpha = tau Gn - u0 Gp,
// with 7 FP32 instructions per epoch beyond the residual.  The Gauss-Newton
// matrix likewise from the nine sums w tau^m g_a g_b (m = 0, 1, 2).
constexpr int kAdjWarps = 16;          // warps (trajectories) per block
constexpr int kAdjEpSmemMax = 6144;    // epochs staged in shared memory

constexpr int kRefineDoubles = 39;     // RefineState, th_cur to H_best

struct AdjTraj {
  TrajC c;
  float cs, sn, u0, dD;  // direction, u0, Delta (FP32)
  double kt, u0d, csd, snd;
  const float4 *quad;    // the trajectory's map (cell table)
};

struct AdjSums {
  float x1, y1, x2, y2;  // sum w r g, sum w r tau g (pixel axes)
  float h[9];            // sum w tau^m g_a g_b: m-major, (xx, xy, yy)
};

template <bool WITH_H>
__device__ __forceinline__ void adj_add(AdjSums &a, float &chi, float w,
                                        float fc, float Ac, float tau,
                                        float gx, float gy, float Fs,
                                        float Bc) {
  const float r = __fsub_rn(fc, __fmaf_rn(Fs, Ac, Bc));
  const float wr = __fmul_rn(w, r);
  chi = __fmaf_rn(wr, r, chi);
  const float wrt = __fmul_rn(wr, tau);
  a.x1 = __fmaf_rn(wr, gx, a.x1);
  a.y1 = __fmaf_rn(wr, gy, a.y1);
  a.x2 = __fmaf_rn(wrt, gx, a.x2);
  a.y2 = __fmaf_rn(wrt, gy, a.y2);
  if (WITH_H) {
    const float wgx = __fmul_rn(w, gx), wgy = __fmul_rn(w, gy);
    const float pxx = __fmul_rn(wgx, gx), pxy = __fmul_rn(wgx, gy);
    const float pyy = __fmul_rn(wgy, gy);
    const float t2 = __fmul_rn(tau, tau);
    a.h[0] = __fadd_rn(a.h[0], pxx);
    a.h[1] = __fadd_rn(a.h[1], pxy);
    a.h[2] = __fadd_rn(a.h[2], pyy);
    a.h[3] = __fmaf_rn(tau, pxx, a.h[3]);
    a.h[4] = __fmaf_rn(tau, pxy, a.h[4]);
    a.h[5] = __fmaf_rn(tau, pyy, a.h[5]);
    a.h[6] = __fmaf_rn(t2, pxx, a.h[6]);
    a.h[7] = __fmaf_rn(t2, pxy, a.h[7]);
    a.h[8] = __fmaf_rn(t2, pyy, a.h[8]);
  }
}

// A - 1, tau and the pixel-axis gradient of an epoch outside the map
// (single lens in u^2 = tau^2 + u0^2, the search's arithmetic for A)
__device__ __forceinline__ float out_point(const AdjTraj &T, float t,
                                           float &tau, float &gx, float &gy) {
  tau = __fmaf_rn(T.c.kt, t, T.c.bt);
  const float u2 = __fmaf_rn(tau, tau, T.c.u02);
  const float rr = rsqrt_approx(__fmul_rn(u2, __fadd_rn(u2, 4.f)));
  const float am1 = __fsub_rn(__fmul_rn(__fadd_rn(u2, 2.f), rr), 1.f);
  // Delta D, D = (dA/du)/u = -8 (u^2 (u^2 + 4))^(-3/2)
  const float dD = __fmul_rn(__fmul_rn(-8.f, T.dD),
                             __fmul_rn(rr, __fmul_rn(rr, rr)));
  const float y1 = __fmaf_rn(tau, T.cs, -__fmul_rn(T.u0, T.sn));
  const float y2 = __fmaf_rn(tau, T.sn, __fmul_rn(T.u0, T.cs));
  gx = __fmul_rn(dD, y1);
  gy = __fmul_rn(dD, y2);
  return am1;
}

// A - 1, tau and the pixel-axis gradient inside the map (the search's
// bilinear lookup; the cell's slopes at (fx, fy))
__device__ __forceinline__ float in_point(const SearchParams &P,
                                          const AdjTraj &T, float t,
                                          float &tau, float &gx, float &gy) {
  const float vx = __fmaf_rn(T.c.ax, t, T.c.bx);
  const float vy = __fmaf_rn(T.c.ay, t, T.c.by);
  tau = __fmaf_rn(T.c.kt, t, T.c.bt);
  TexPos p;
  if (!tex_pos(P, vx, vy, p)) {
    gx = gy = 0.f;
    return 0.f;
  }
  const float4 q = __ldg(&P.quad[p.idx]);
  const float r0 = __fmaf_rn(p.fx, q.y, q.x);
  const float dr = __fmaf_rn(p.fx, q.w, q.z);
  gx = __fmaf_rn(p.fy, q.w, q.y);
  gy = dr;
  return __fmaf_rn(p.fy, dr, r0);
}

__device__ __forceinline__ float warp_sum_f32(float x) {
#pragma unroll
  for (int o = 16; o; o >>= 1) x = __fadd_rn(x, __shfl_xor_sync(kFull, x, o));
  return x;
}

// constants of theta = (t0, tE, u0, alpha), t0 absolute
__device__ __forceinline__ AdjTraj adj_traj(const SearchParams &P,
                                            const Epochs &ep,
                                            const double *th, double t_ref,
                                            const float4 *quad) {
  const double t0 = th[0], tE = th[1];
  const double u0 = th[2], al = th[3];
  double sn, cs;
  sincos(al, &sn, &cs);
  const double tEc = (tE > 1e-6) ? tE : 1e-6;  // the host rejects tE <= 0
  double tlo, thi;
  slab_tau(P.L, u0, cs, sn, tlo, thi);
  AdjTraj T;
  T.c = make_traj(P, ep, u0, cs, sn, t0 - t_ref, 1.0 / (tEc * P.dlt), tEc,
                  tlo, thi);
  T.cs = (float)cs;
  T.sn = (float)sn;
  T.u0 = (float)u0;
  T.dD = P.dltf;
  T.kt = 1.0 / tEc;
  T.u0d = u0;
  T.csd = cs;
  T.snd = sn;
  T.quad = quad;
  return T;
}

// sweep 2 of one warp: residuals, chi^2 and the gradient (and Gauss-Newton)
// sums, across lanes (chi^2 in FP64, as the search's phase 2; the rest FP32)
template <bool WITH_H, int UN>
__device__ __forceinline__ double adj_sweep(const SearchParams &Q,
                                            const Epochs &ep,
                                            const AdjTraj &T, float fFs,
                                            float fBc, int lane,
                                            AdjSums &a) {
  a.x1 = a.y1 = a.x2 = a.y2 = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) a.h[k] = 0.f;
  float chi = 0.f;
#pragma unroll 2
  for (int e = lane_start(0, lane); e < T.c.e_in; e += 32) {
    const float2 v = ep.tw[e];
    float tau, gx, gy;
    const float Ac = out_point(T, v.x, tau, gx, gy);
    adj_add<WITH_H>(a, chi, v.y, ep.fc[e], Ac, tau, gx, gy, fFs, fBc);
  }
#pragma unroll UN
  for (int e = lane_start(T.c.e_in, lane); e < T.c.e_out; e += 32) {
    const float2 v = ep.tw[e];
    float tau, gx, gy;
    const float Ac = in_point(Q, T, v.x, tau, gx, gy);
    adj_add<WITH_H>(a, chi, v.y, ep.fc[e], Ac, tau, gx, gy, fFs, fBc);
  }
#pragma unroll 2
  for (int e = lane_start(T.c.e_out, lane); e < Q.n_ep; e += 32) {
    const float2 v = ep.tw[e];
    float tau, gx, gy;
    const float Ac = out_point(T, v.x, tau, gx, gy);
    adj_add<WITH_H>(a, chi, v.y, ep.fc[e], Ac, tau, gx, gy, fFs, fBc);
  }
  double x = (double)chi;
#pragma unroll
  for (int o = 16; o; o >>= 1) x = __dadd_rn(x, __shfl_xor_sync(kFull, x, o));
  a.x1 = warp_sum_f32(a.x1);
  a.y1 = warp_sum_f32(a.y1);
  a.x2 = warp_sum_f32(a.x2);
  a.y2 = warp_sum_f32(a.y2);
  if (WITH_H) {
#pragma unroll
    for (int k = 0; k < 9; ++k) a.h[k] = warp_sum_f32(a.h[k]);
  }
  return x;
}

// chi^2, gradient (4) and Gauss-Newton matrix (10, upper triangle,
// row-major) of one trajectory from its sums; outputs may be null
template <bool WITH_H>
__device__ __forceinline__ void adj_assemble(const SearchParams &P,
                                             const AdjTraj &Tj,
                                             const AdjSums &a, double fs,
                                             double x2, double *chi2,
                                             double *grad, double *h) {
  const double c = Tj.csd, s = Tj.snd, u0 = Tj.u0d, kt = Tj.kt;
  const double iD = P.invD;
  const double P1 = (c * a.x1 + s * a.y1) * iD;
  const double N1 = (c * a.y1 - s * a.x1) * iD;
  const double P2 = (c * a.x2 + s * a.y2) * iD;
  const double N2 = (c * a.y2 - s * a.x2) * iD;
  if (chi2) *chi2 = isnan(x2) ? CUDART_INF : x2;
  if (grad) {
    const double m2 = -2.0 * fs;
    grad[0] = m2 * (-kt * P1);
    grad[1] = m2 * (-kt * P2);
    grad[2] = m2 * N1;
    grad[3] = m2 * (N2 - u0 * P1);
  }
  if (WITH_H && h) {
    const double d2 = iD * iD, f2 = fs * fs;
    double spp[3], spn[3], snn[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double xx = a.h[3 * m], xy = a.h[3 * m + 1], yy = a.h[3 * m + 2];
      spp[m] = (c * c * xx + 2.0 * c * s * xy + s * s * yy) * d2;
      snn[m] = (s * s * xx - 2.0 * c * s * xy + c * c * yy) * d2;
      spn[m] = (c * s * (yy - xx) + (c * c - s * s) * xy) * d2;
    }
    h[0] = f2 * kt * kt * spp[0];
    h[1] = f2 * kt * kt * spp[1];
    h[2] = f2 * -kt * spn[0];
    h[3] = f2 * -kt * (spn[1] - u0 * spp[0]);
    h[4] = f2 * kt * kt * spp[2];
    h[5] = f2 * -kt * spn[1];
    h[6] = f2 * -kt * (spn[2] - u0 * spp[1]);
    h[7] = f2 * snn[0];
    h[8] = f2 * (snn[1] - u0 * spn[0]);
    h[9] = f2 * (snn[2] - 2.0 * u0 * spn[1] + u0 * u0 * spp[0]);
  }
}

// theta_i = (t0, tE, u0, alpha) with absolute t0, on the map P.quad or,
// when tq is set, on the map tq[i] (maps of one geometry).  Outputs (any
// may be null): chi2[i], grad[4 i + k], Fs[i], Fb[i], flags[i].
// MINB: blocks per SM, UN: inside-map epochs in flight per lane (adj_split).
template <bool EP_SMEM, int MINB, int UN>
__global__ void __launch_bounds__(kAdjWarps * 32, MINB)
    k_theta(const SearchParams P, const double *__restrict__ theta,
            const float4 *const *__restrict__ tq, int n, double t_ref,
            double *chi2, double *grad, double *Fs, double *Fb, int *flags) {
  extern __shared__ __align__(16) float4 s_ep[];
  __shared__ AdjTraj s_tr[kAdjWarps];
  __shared__ Acc s_acc[kAdjWarps];
  __shared__ double s_Fs[kAdjWarps], s_Bc[kAdjWarps];
  __shared__ int s_deg[kAdjWarps];
  __shared__ AdjSums s_sum[kAdjWarps];
  __shared__ double s_chi[kAdjWarps];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int i0 = blockIdx.x * kAdjWarps;
  const int i = i0 + warp;
  if (EP_SMEM)
    for (int e = threadIdx.x; e < P.n_ep; e += blockDim.x) s_ep[e] = P.ep[e];
  // set-up, one lane per trajectory (the epoch ranges from the global copy:
  // the shared one is still being written)
  if (warp == 0 && lane < kAdjWarps && i0 + lane < n) {
    const int j = i0 + lane;
    s_tr[lane] = adj_traj(P, epochs_at(P.ep, P.n_ep), theta + 4 * j, t_ref,
                          tq ? tq[j] : P.quad);
  }
  __syncthreads();
  const Epochs ep = epochs_at(EP_SMEM ? s_ep : P.ep, P.n_ep);
  const bool live = i < n;
  AdjTraj T;
  if (live) T = s_tr[warp];
  SearchParams Q = P;  // this warp's map
  Q.quad = live ? T.quad : P.quad;
  // sweep 1: the normal-equation sums (the search's phase 1)
  if (live) {
    const Acc a = phase1<false, 0, UN>(Q, ep, T.c, lane);
    if (lane == 0) s_acc[warp] = a;
  }
  __syncthreads();
  if (warp == 0 && lane < kAdjWarps && i0 + lane < n) {
    const Acc a = s_acc[lane];
    const Fit2 f = fit2(P, (double)a.a, (double)a.b, (double)a.d);
    s_Fs[lane] = f.Fs;
    s_Bc[lane] = f.Bc;
    s_deg[lane] = f.degenerate ? 1 : 0;
  }
  __syncthreads();
  // sweep 2: residuals, chi^2 and the gradient (and Gauss-Newton) sums
  if (live) {
    const float fFs = __double2float_rn(s_Fs[warp]);
    const float fBc = __double2float_rn(s_Bc[warp]);
    AdjSums a;
    const double x =
        adj_sweep<false, UN>(Q, ep, T, fFs, fBc, lane, a);
    if (lane == 0) {
      s_chi[warp] = x;
      s_sum[warp] = a;
    }
  }
  __syncthreads();
  // assembly of the outputs, one lane per trajectory
  if (warp == 0 && lane < kAdjWarps && i0 + lane < n) {
    const int j = i0 + lane;
    const double fs = s_Fs[lane];
    adj_assemble<false>(P, s_tr[lane], s_sum[lane], fs, s_chi[lane],
                        chi2 ? chi2 + j : nullptr,
                        grad ? grad + 4 * (size_t)j : nullptr, nullptr);
    if (Fs) Fs[j] = fs;
    if (Fb) Fb[j] = s_Bc[lane] + P.Fref - fs;
    if (flags) flags[j] = s_deg[lane] ? MORSE_FIT_DEGENERATE : 0;
  }
}

// Solve (H + lam diag(H) + eps I) x = b for a 4x4 symmetric H given as its
// upper triangle; Cholesky in FP64.  Returns false if not positive definite.
__device__ bool lm_solve(const double *h, double lam, const double *b,
                         double *x) {
  double M[4][4];
  int m = 0;
  for (int k = 0; k < 4; ++k)
    for (int l = k; l < 4; ++l) {
      M[k][l] = M[l][k] = h[m];
      ++m;
    }
  for (int k = 0; k < 4; ++k) M[k][k] = M[k][k] * (1.0 + lam) + 1e-300;
  double L[4][4] = {{0}};
  for (int j = 0; j < 4; ++j) {
    double sum = M[j][j];
    for (int k = 0; k < j; ++k) sum -= L[j][k] * L[j][k];
    if (!(sum > 0.0)) return false;
    L[j][j] = sqrt(sum);
    for (int i2 = j + 1; i2 < 4; ++i2) {
      double t = M[i2][j];
      for (int k = 0; k < j; ++k) t -= L[i2][k] * L[j][k];
      L[i2][j] = t / L[j][j];
    }
  }
  double y[4];
  for (int i2 = 0; i2 < 4; ++i2) {
    double t = b[i2];
    for (int k = 0; k < i2; ++k) t -= L[i2][k] * y[k];
    y[i2] = t / L[i2][i2];
  }
  for (int i2 = 3; i2 >= 0; --i2) {
    double t = y[i2];
    for (int k = i2 + 1; k < 4; ++k) t -= L[k][i2] * x[k];
    x[i2] = t / L[i2][i2];
  }
  return true;
}

__device__ __forceinline__ bool same_traj(const TrajC &a, const TrajC &b) {
  return __float_as_int(a.ax) == __float_as_int(b.ax) &&
         __float_as_int(a.bx) == __float_as_int(b.bx) &&
         __float_as_int(a.ay) == __float_as_int(b.ay) &&
         __float_as_int(a.by) == __float_as_int(b.by) &&
         __float_as_int(a.kt) == __float_as_int(b.kt) &&
         __float_as_int(a.bt) == __float_as_int(b.bt) &&
         __float_as_int(a.u02) == __float_as_int(b.u02) &&
         a.e_in == b.e_in && a.e_out == b.e_out;
}

// One Levenberg-Marquardt step of trajectory i (one thread).  The
// evaluation at theta_cur is accepted if it lowered chi^2 (damping / 3) or
// rejected (damping x 4, back to theta_best); then the next point is
// theta_best - (H + lam diag H)^-1 g at the best point.
__device__ __forceinline__ void lm_step(const RefineState &S, int i) {
  double lam = S.lam[i];
  const double c = S.chi2_cur[i];
  if (c < S.chi2_best[i]) {
    S.chi2_best[i] = c;
    for (int k = 0; k < 4; ++k) {
      S.th_best[4 * i + k] = S.th_cur[4 * i + k];
      S.g_best[4 * i + k] = S.g_cur[4 * i + k];
    }
    for (int k = 0; k < 10; ++k) S.H_best[10 * i + k] = S.H_cur[10 * i + k];
    lam = fmax(lam / 3.0, 1e-12);
  } else {
    lam = fmin(lam * 4.0, 1e12);
  }
  double neg_g[4], dx[4] = {0, 0, 0, 0};
  for (int k = 0; k < 4; ++k) neg_g[k] = -S.g_best[4 * i + k];
  bool ok = false;
  for (int tries = 0; tries < 8 && !ok; ++tries) {
    ok = lm_solve(S.H_best + 10 * i, lam, neg_g, dx);
    if (!ok) lam = fmin(lam * 10.0, 1e12);
  }
  if (!ok)
    for (int k = 0; k < 4; ++k) dx[k] = 0.0;
  S.lam[i] = lam;
  for (int k = 0; k < 4; ++k)
    S.th_cur[4 * i + k] = S.th_best[4 * i + k] + dx[k];
  // keep tE positive
  const double tE = S.th_cur[4 * i + 1];
  const double tEb = S.th_best[4 * i + 1];
  if (!(tE > 0.05 * tEb)) S.th_cur[4 * i + 1] = 0.5 * tEb;
}

// All iterations of the refinement of kAdjWarps trajectories in one launch:
// their states stay in shared memory, the light curve is staged once.
//
// A point whose track constants (the FP32 set that both sweeps use) are
// those of the best point has the best point's chi^2 bit for bit and is
// rejected whatever its gradient: its sweeps are not taken.  With the
// damping at its ceiling such a step repeats for ever, and a block whose
// trajectories all do so ends.
//
// With one launch per evaluation and one per step an iteration of 2047
// trajectories of 3000 epochs took 59 us, here 40 (81k cycles):
// the two sweeps 46k, of which 33k are the L1 gather rate, and 34k the chain
// of FP64 set-up, fit, assembly and step that one warp runs for all 16; with
// one trajectory per SM 29 us, 27k and 34k.  Two blocks of 8 warps or four of
// 4 per SM were the same or slower: their FP64 chains share the SM's pipe.
//
// The chain costs the same for 32 trajectories, its lanes, as for 16: where
// there are more than one wave of blocks and the sweeps are short, a warp
// takes TPW = 2 trajectories (launch_refine).
template <bool EP_SMEM, int MINB, int UN, int TPW>
__global__ void __launch_bounds__(kAdjWarps * 32, MINB)
    k_refine(const SearchParams P, RefineState S,
             const float4 *const *__restrict__ tq, int n, int iters,
             double t_ref) {
  extern __shared__ __align__(16) float4 s_ep[];
  constexpr int kTr = kAdjWarps * TPW;  // trajectories of a block, at most
  __shared__ AdjTraj s_tr[kTr];
  __shared__ TrajC s_best[kTr];
  __shared__ Acc s_acc[kTr];
  __shared__ double s_Fs[kTr], s_Bc[kTr];
  __shared__ AdjSums s_sum[kTr];
  __shared__ double s_chi[kTr];
  __shared__ double s_state[kTr * kRefineDoubles];
  __shared__ int s_eval[kTr], s_more;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int warps = blockDim.x >> 5;
  const int i0 = blockIdx.x * warps * TPW;
  const bool mine = warp == 0 && lane < warps * TPW && i0 + lane < n;
  if (EP_SMEM)
    for (int e = threadIdx.x; e < P.n_ep; e += blockDim.x) s_ep[e] = P.ep[e];
  // the block's states (each read and written by one lane of warp 0 only)
  RefineState B;
  B.th_cur = s_state;
  B.th_best = B.th_cur + 4 * kTr;
  B.chi2_cur = B.th_best + 4 * kTr;
  B.chi2_best = B.chi2_cur + kTr;
  B.lam = B.chi2_best + kTr;
  B.g_cur = B.lam + kTr;
  B.g_best = B.g_cur + 4 * kTr;
  B.H_cur = B.g_best + 4 * kTr;
  B.H_best = B.H_cur + 10 * kTr;
  const float4 *quad = P.quad;
  if (mine) {
    const int j = i0 + lane;
    for (int k = 0; k < 4; ++k) {
      B.th_cur[4 * lane + k] = S.th_cur[4 * j + k];
      B.th_best[4 * lane + k] = S.th_best[4 * j + k];
      B.g_best[4 * lane + k] = 0.0;
    }
    for (int k = 0; k < 10; ++k) B.H_best[10 * lane + k] = 0.0;
    B.chi2_best[lane] = S.chi2_best[j];
    B.lam[lane] = S.lam[j];
    if (tq) quad = tq[j];
  }
  __syncthreads();
  const Epochs ep = epochs_at(EP_SMEM ? s_ep : P.ep, P.n_ep);
  for (int it = 0; it < iters; ++it) {
    if (mine) {
      const AdjTraj T = adj_traj(P, ep, B.th_cur + 4 * lane, t_ref, quad);
      s_tr[lane] = T;
      s_eval[lane] = !(B.chi2_best[lane] < CUDART_INF) ||
                     !same_traj(T.c, s_best[lane]);
    }
    __syncthreads();
    AdjTraj T;
    SearchParams Q = P;  // the trajectory's map
    bool eval = false;
#pragma unroll 1
    for (int r = 0; r < TPW; ++r) {
      const int k = warp + r * warps;
      eval = i0 + k < n && s_eval[k];
      if (eval) {
        T = s_tr[k];
        Q.quad = T.quad;
        const Acc a = phase1<false, 0, UN>(Q, ep, T.c, lane);
        if (lane == 0) s_acc[k] = a;
      }
    }
    __syncthreads();
    if (mine && s_eval[lane]) {
      const Acc a = s_acc[lane];
      const Fit2 f = fit2(P, (double)a.a, (double)a.b, (double)a.d);
      s_Fs[lane] = f.Fs;
      s_Bc[lane] = f.Bc;
    }
    __syncthreads();
#pragma unroll 1
    for (int r = 0; r < TPW; ++r) {
      const int k = warp + r * warps;
      if (TPW > 1) {
        eval = i0 + k < n && s_eval[k];
        if (eval) T = s_tr[k];
        Q.quad = T.quad;
      }
      if (eval) {
        AdjSums a;
        const double x =
            adj_sweep<true, UN>(Q, ep, T, __double2float_rn(s_Fs[k]),
                                __double2float_rn(s_Bc[k]), lane, a);
        if (lane == 0) {
          s_chi[k] = x;
          s_sum[k] = a;
        }
      }
    }
    __syncthreads();
    if (warp == 0) {
      bool more = false;
      if (mine) {
        const bool better = s_eval[lane] && s_chi[lane] < B.chi2_best[lane];
        if (s_eval[lane])
          adj_assemble<true>(P, s_tr[lane], s_sum[lane], s_Fs[lane],
                             s_chi[lane], B.chi2_cur + lane,
                             B.g_cur + 4 * lane, B.H_cur + 10 * lane);
        else
          B.chi2_cur[lane] = B.chi2_best[lane];
        more = s_eval[lane] || B.lam[lane] < 1e12;
        if (more) lm_step(B, lane);
        if (better) s_best[lane] = s_tr[lane].c;
      }
      more = __any_sync(kFull, more);
      if (lane == 0) s_more = more;
    }
    __syncthreads();
    if (!s_more) break;
  }
  if (mine)
    for (int k = 0; k < 4; ++k)
      S.th_best[4 * (i0 + lane) + k] = B.th_best[4 * lane + k];
}

__global__ void k_lm_init(RefineState S, const morse_fit *starts, int n,
                          double lam0) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const morse_fit f = starts[i];
  S.th_cur[4 * i + 0] = f.t0;
  S.th_cur[4 * i + 1] = f.tE;
  S.th_cur[4 * i + 2] = f.u0;
  S.th_cur[4 * i + 3] = f.alpha;
  for (int k = 0; k < 4; ++k) S.th_best[4 * i + k] = S.th_cur[4 * i + k];
  S.chi2_best[i] = CUDART_INF;
  S.lam[i] = lam0;
}

// records of the refined trajectories: theta_best, its chi^2 and fluxes
__global__ void k_lm_finish(RefineState S, const morse_fit *starts, int n,
                            morse_fit *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  morse_fit f;
  f.t0 = S.th_best[4 * i + 0];
  f.tE = S.th_best[4 * i + 1];
  f.u0 = S.th_best[4 * i + 2];
  f.alpha = S.th_best[4 * i + 3];
  f.chi2 = S.chi2_cur[i];
  f.Fs = S.Fs[i];
  f.Fb = S.Fb[i];
  f.idx = starts[i].idx;
  f.flags = S.flags[i] | MORSE_FIT_REFINED;
  f.reserved = 0;
  out[i] = f;
}

}  // namespace

// The form of the evaluation kernels for a number of blocks.  Up to one per
// SM a thread may take 128 registers, for eight texel gathers in flight per
// lane; above, two blocks per SM and four gathers.
// 2047 trajectories of 3000 epochs: 42 -> 36 us an evaluation; with more
// blocks than SMs a second wave would cost more (refinement of 4096: 3.2 ms
// against twice 2.0).
template <typename... A>
static void run_theta(const SearchParams &P, int n, int sm_count,
                      cudaStream_t st, A... args) {
  const int blocks = (n + kAdjWarps - 1) / kAdjWarps;
  const int threads = kAdjWarps * 32;
  const bool few = blocks <= sm_count;
  const size_t sh = sizeof(float4) * P.n_ep;
  if (P.n_ep <= kAdjEpSmemMax) {
    if (few)
      k_theta<true, 1, 8><<<blocks, threads, sh, st>>>(P, args...);
    else
      k_theta<true, 2, 4><<<blocks, threads, sh, st>>>(P, args...);
  } else {
    if (few)
      k_theta<false, 1, 8><<<blocks, threads, 0, st>>>(P, args...);
    else
      k_theta<false, 2, 4><<<blocks, threads, 0, st>>>(P, args...);
  }
}

template <typename K>
static cudaError_t ep_smem(K kernel) {
  return cudaFuncSetAttribute(kernel,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(sizeof(float4) * kAdjEpSmemMax));
}

cudaError_t adjoint_setup() {
  cudaError_t e = ep_smem(k_theta<true, 1, 8>);
  if (e == cudaSuccess) e = ep_smem(k_theta<true, 2, 4>);
  if (e == cudaSuccess) e = ep_smem(k_refine<true, 1, 8, 1>);
  if (e == cudaSuccess) e = ep_smem(k_refine<true, 2, 4, 1>);
  if (e == cudaSuccess) e = ep_smem(k_refine<true, 2, 4, 2>);
  return e;
}

cudaError_t launch_theta(const SearchParams &P, const double *theta, int n,
                         double t_ref, double *chi2, double *grad, double *Fs,
                         double *Fb, int *flags, int sm_count,
                         cudaStream_t st, const float4 *const *tq) {
  if (n <= 0) return cudaSuccess;
  run_theta(P, n, sm_count, st, theta, tq, n, t_ref, chi2, grad, Fs, Fb, flags);
  return cudaGetLastError();
}

// Blocks of as many warps as spread the trajectories over the SMs, at most
// kAdjWarps; two trajectories to a warp for light curves of up to
// kRefinePairEpMax epochs where one to a warp would take more than two blocks
// per SM.  20 iterations of 4865, 9728, 9800 and 20 000 starts: 64 epochs 856,
// 961, 1329, 2264 -> 544, 624, 1065, 1640 us, 1500 epochs 1308, 1722, 2301,
// 3906 -> 1134, 1379, 2255, 3525; 2000 epochs 1443, 1954, 2590, 4440 against
// 1333, 1624, 2645, 4152 and 4000 epochs 2006, 2958, 3833, 6612 against 2106,
// 2644, 4216, 6631: the last block's sweeps are twice as long.
constexpr int kRefinePairEpMax = 1536;
cudaError_t launch_refine(const SearchParams &P, const RefineState &S, int n,
                          int iters, double t_ref, int sm_count,
                          cudaStream_t st, const float4 *const *tq) {
  if (n <= 0 || iters <= 0) return cudaSuccess;
  const int warps = std::min(kAdjWarps, (n + sm_count - 1) / sm_count);
  const int blocks = (n + warps - 1) / warps, threads = 32 * warps;
  const bool few = blocks <= sm_count;
  const size_t sh = sizeof(float4) * P.n_ep;
  if (P.n_ep <= kRefinePairEpMax && blocks > 2 * sm_count)
    k_refine<true, 2, 4, 2><<<(blocks + 1) / 2, threads, sh, st>>>(
        P, S, tq, n, iters, t_ref);
  else if (P.n_ep <= kAdjEpSmemMax && few)
    k_refine<true, 1, 8, 1><<<blocks, threads, sh, st>>>(P, S, tq, n, iters,
                                                          t_ref);
  else if (P.n_ep <= kAdjEpSmemMax)
    k_refine<true, 2, 4, 1><<<blocks, threads, sh, st>>>(P, S, tq, n, iters,
                                                          t_ref);
  else if (few)
    k_refine<false, 1, 8, 1><<<blocks, threads, 0, st>>>(P, S, tq, n, iters,
                                                          t_ref);
  else
    k_refine<false, 2, 4, 1><<<blocks, threads, 0, st>>>(P, S, tq, n, iters,
                                                          t_ref);
  return cudaGetLastError();
}

cudaError_t launch_lm_init(const RefineState &S, const morse_fit *starts,
                           int n, double lam0, cudaStream_t st) {
  k_lm_init<<<(n + 127) / 128, 128, 0, st>>>(S, starts, n, lam0);
  return cudaGetLastError();
}

cudaError_t launch_lm_finish(const RefineState &S, const morse_fit *starts,
                             int n, morse_fit *out, cudaStream_t st) {
  k_lm_finish<<<(n + 127) / 128, 128, 0, st>>>(S, starts, n, out);
  return cudaGetLastError();
}

}  // namespace morse
