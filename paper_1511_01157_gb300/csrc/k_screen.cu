// Screening of the trajectory grid search: which trajectories can enter the
// top-K at all.
//
// chi^2 is a sum of non-negative terms, so the smallest chi^2 that any flux
// fit gives on a subset of the epochs bounds the chi^2 of the whole light
// curve from below (screen_lb).  Each event keeps small subsets, drawn in
// proportion to the epochs' information w (F - F_mean)^2
// (morse_event_create): on a config-1 event (3000 epochs) the bounds of 64
// such epochs exceed the final K-th chi^2 for 94 % of the grid's
// trajectories, where 64 evenly spaced epochs discard 64 %.
//
//   k_screen       the bound of every trajectory on the smallest subset,
//                  kept as a 16-bit code, and a histogram of the codes
//   k_pilot_list   the trajectories of lowest bound
//   k_pilot        upper bounds of their chi^2 over the whole light curve
//   k_list         the K-th of those, a rigorous threshold near the final
//                  one, and the list of trajectories at or below it
//
// The listed search (k_search_list) then runs over the list alone, with the
// larger subsets first.  Results are those of the unscreened search bit for
// bit: a discarded trajectory's chi^2 exceeds K others', and every listed
// one is evaluated by the same device functions.  Measured, call by call
// (1024^2 map, 1.44 M trajectories, 3000 epochs, K = 256): 3.25 -> 0.84 ms;
// four maps of a sweep 13.5 -> 2.95 ms.  The host screens from 16 384
// trajectories and 128 epochs on; below that a search is bound by its
// launches and its latency, and there are too few trajectories to rank.
// Where more than half of the grid stays on the list (light curves of weak
// signal), the whole range is searched as before (k_search), the screening
// costing a share 64 / n_epochs.
#ifndef MORSE_PK_ASM
#define MORSE_PK_ASM 1
#endif
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include <algorithm>

#include "morse_internal.cuh"
#include "search_common.cuh"

namespace morse {

namespace {

using namespace dev;

constexpr int kScreenThreads = 256;
constexpr int kScreenMax = 128;  // epochs of the smallest subset, at most

// Two trajectories per lane (32 apart, packed FP32), every lane over the
// whole subset: no reductions, one broadcast shared load of an epoch for 64
// trajectories, and a warp's gathers fall on one or two lines of the map.
template <bool H>
__global__ void __launch_bounds__(kScreenThreads)
    k_screen(const SearchParams P, const ScreenBufs B) {
  __shared__ float4 s_ep[kScreenMax];
  __shared__ unsigned s_hist[kScreenBins];
  const ScreenLv V = P.lv[0];
  const Epochs ep = epochs_at(V.ep, V.m);
  for (int e = threadIdx.x; e < V.m; e += blockDim.x)
    s_ep[e] = make_float4(ep.tw[e].x, ep.tw[e].y, ep.wf[e], 0.f);
  for (int b = threadIdx.x; b < kScreenBins; b += blockDim.x) s_hist[b] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned n = (unsigned)P.count;
  const unsigned step = gridDim.x * (kScreenThreads / 32) * 64u;
  for (unsigned i0 = (blockIdx.x * (kScreenThreads / 32) +
                      (threadIdx.x >> 5)) * 64u;
       i0 < n; i0 += step) {
    const unsigned ia = i0 + lane, ib = ia + 32;
    const unsigned ja = (unsigned)P.first + min(ia, n - 1);
    const unsigned jb = (unsigned)P.first + min(ib, n - 1);
    double xi, xo;
    const TrajC ca = traj_base_of(P, ja, xi, xo);
    const float ain = __double2float_rd(xi), aout = __double2float_ru(xo);
    const TrajC cb = traj_base_of(P, jb, xi, xo);
    const float bin = __double2float_rd(xi), bout = __double2float_ru(xo);
    const TrajP c = pack_traj(ca, cb);
    Acc2 s = {f2(0.f), f2(0.f), f2(0.f)};
#pragma unroll 4
    for (int e = 0; e < V.m; ++e) {
      const float4 v = s_ep[e];
      const float2 tt = f2(v.x);
      const bool ina = v.x > ain && v.x < aout;
      const bool inb = v.x > bin && v.x < bout;
      float2 Ac = make_float2(0.f, 0.f);
      if (ina || inb) {
        const float2 vx = pk_fma(c.ax, tt, c.bx);
        const float2 vy = pk_fma(c.ay, tt, c.by);
        // (outside: any cell of the map, the value is not used)
        const float xa = ina ? vx.x : 0.f, ya = ina ? vy.x : 0.f;
        const float xb = inb ? vx.y : 0.f, yb = inb ? vy.y : 0.f;
        Ac.x = H ? bilinear_h_m1(P, xa, ya) : bilinear_m1(P, xa, ya);
        Ac.y = H ? bilinear_h_m1(P, xb, yb) : bilinear_m1(P, xb, yb);
      }
      if (!ina || !inb) {
        const float2 o = mag2_out_m1(c, tt);
        if (!ina) Ac.x = o.x;
        if (!inb) Ac.y = o.y;
      }
      acc2_add(s, f2(v.y), f2(v.z), Ac);
    }
    const Acc sa = {s.a.x, s.b.x, s.d.x}, sb = {s.a.y, s.b.y, s.d.y};
    unsigned ka = __float_as_uint(screen_lb(V, sa)) >> 16;
    unsigned kb = __float_as_uint(screen_lb(V, sb)) >> 16;
    if (P.linemax) {  // trajectories of cut lines are not searched
      const unsigned line = (unsigned)P.line;
      if (__ldg(&P.linemax[ja / line]) < P.a_min) ka = kScreenCut;
      if (__ldg(&P.linemax[jb / line]) < P.a_min) kb = kScreenCut;
    }
    if (ia < n) {
      B.code[ia] = (unsigned short)ka;
      if (ka != kScreenCut) atomicAdd(&s_hist[ka >> 3], 1u);
    }
    if (ib < n) {
      B.code[ib] = (unsigned short)kb;
      if (kb != kScreenCut) atomicAdd(&s_hist[kb >> 3], 1u);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kScreenBins; b += blockDim.x)
    if (s_hist[b]) atomicAdd(&B.hist[b], s_hist[b]);
}

// Appends the trajectories keep() accepts to out[], in ascending order
// within a block's chunks of codes (one atomic per chunk): neighbouring
// entries mostly share a line of the map.
template <typename Keep>
__device__ __forceinline__ void append(const ScreenBufs &B, unsigned n,
                                       unsigned cap, unsigned *out,
                                       unsigned *len, const Keep &keep) {
  constexpr int kPer = 8;  // codes per thread: one 16-byte load
  __shared__ unsigned s_w[32], s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  const unsigned chunk = blockDim.x * kPer;
  for (unsigned c0 = blockIdx.x * chunk; c0 < n; c0 += gridDim.x * chunk) {
    const unsigned i0 = c0 + threadIdx.x * kPer;
    unsigned m = 0;
    if (i0 < n) {
      const uint4 q = *reinterpret_cast<const uint4 *>(B.code + i0);
      const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const unsigned code = (w[k >> 1] >> (16 * (k & 1))) & 0xFFFFu;
        if (i0 + k < n && code != kScreenCut && keep(code, i0 + k))
          m |= 1u << k;
      }
    }
    const unsigned c = __popc(m);
    unsigned p = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned v = __shfl_up_sync(kFull, p, o);
      if (lane >= o) p += v;
    }
    if (lane == 31) s_w[warp] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned t = 0;
      for (int k = 0; k < nw; ++k) {
        const unsigned v = s_w[k];
        s_w[k] = t;
        t += v;
      }
      s_base = t ? atomicAdd(len, t) : 0u;
    }
    __syncthreads();
    unsigned at = s_base + s_w[warp] + p - c;
    for (; m; m &= m - 1, ++at)
      if (at < cap) out[at] = i0 + (__ffs(m) - 1);
    __syncthreads();
  }
}

// The pilot's list: every trajectory below the histogram bin that holds the
// want-th lowest code, and a hashed sample of that bin's (codes are equal
// there as far as the histogram tells: all of them, where the bounds say
// nothing).
__global__ void __launch_bounds__(256)
    k_pilot_list(const SearchParams P, const ScreenBufs B) {
  __shared__ unsigned s_sum[256], s_cut, s_r;
  constexpr int kPer = kScreenBins / 256;
  unsigned t = 0;
  for (int k = 0; k < kPer; ++k) t += B.hist[threadIdx.x * kPer + k];
  s_sum[threadIdx.x] = t;
  if (threadIdx.x == 0) {
    s_cut = kScreenBins;
    s_r = 1;
  }
  __syncthreads();
  for (int o = 1; o < 256; o <<= 1) {
    const unsigned v = threadIdx.x >= o ? s_sum[threadIdx.x - o] : 0u;
    __syncthreads();
    s_sum[threadIdx.x] += v;
    __syncthreads();
  }
  unsigned below = s_sum[threadIdx.x] - t;
  if (below < B.want && s_sum[threadIdx.x] >= B.want) {
    for (int k = 0; k < kPer; ++k) {
      const unsigned h = B.hist[threadIdx.x * kPer + k];
      if (below + h >= B.want) {
        const unsigned left = B.want - below;
        s_cut = threadIdx.x * kPer + k;
        s_r = (h + left - 1) / left;
        break;
      }
      below += h;
    }
  }
  __syncthreads();
  const unsigned cut = s_cut, r = s_r;
  append(B, (unsigned)P.count, B.pilot_cap, B.pilot, &B.n[0],
         [=](unsigned code, unsigned i) {
           const unsigned b = code >> 3;
           return b < cut ||
                  (b == cut && ((i * 0x9E3779B1u) >> 8) % r == 0u);
         });
}

// Upper bounds of the pilot's chi^2 over the whole light curve (the same
// sums and solve as the search; chi2_upper).  Groups of kPilotTpg entries
// per warp: the FP64 solve of a warp costs the same for 1 and 32
// trajectories, the sweeps grow with their number.
constexpr int kPilotTpg = 4, kPilotWarps = 4;

template <bool STAGED, bool H>
__global__ void __launch_bounds__(kPilotWarps * 32)
    k_pilot(const SearchParams P, const ScreenBufs B) {
  extern __shared__ __align__(16) unsigned char smem[];
  const unsigned n = min(B.n[0], B.pilot_cap);
  const int lane = threadIdx.x & 31;
  const unsigned g0 = (blockIdx.x * kPilotWarps + (threadIdx.x >> 5)) *
                      kPilotTpg;
  if (blockIdx.x * kPilotWarps * kPilotTpg >= n) return;  // whole block
  const float4 *blk = P.ep;
  if (STAGED) {
    float4 *s = reinterpret_cast<float4 *>(smem);
    for (int e = threadIdx.x; e < P.n_ep; e += blockDim.x) s[e] = P.ep[e];
    __syncthreads();
    blk = s;
  }
  const Epochs ep = epochs_at(blk, P.n_ep);
  if (g0 >= n) return;
  const int nv = (int)min((unsigned)kPilotTpg, n - g0);
  const unsigned j = (unsigned)P.first + B.pilot[g0 + (lane < nv ? lane : 0)];
  double xi, xo;
  TrajC mine = traj_base_of(P, j, xi, xo);
  traj_range(ep, P.n_ep, xi, xo, mine);
  Acc ms = {0.f, 0.f, 0.f};
  for (int k = 0; k < nv; k += 2) {
    const int k2 = min(k + 1, nv - 1);
    const TrajC ca = shfl_traj(mine, k), cb = shfl_traj(mine, k2);
    Acc ra, rb;
    phase1_pair<H>(P, ep, ca, cb, lane, ra, rb);
    if (lane == k) ms = ra;
    else if (lane == k2) ms = rb;
  }
  const Fit2 f = fit2(P, (double)ms.a, (double)ms.b, (double)ms.d);
  const double ub =
      chi2_upper(P, (double)ms.a, (double)ms.b, (double)ms.d,
                 (double)__double2float_rn(f.Fs),
                 (double)__double2float_rn(f.Bc));
  if (lane < nv) B.ub[g0 + lane] = fmaxf(__double2float_ru(ub), 0.f);
}

// The threshold: the top_k-th smallest of the pilot's bounds (K distinct
// trajectories have chi^2 at or below it), by four passes of eight bits
// over the FP32 bit patterns, every block for itself; then the list.
__global__ void __launch_bounds__(256)
    k_list(const SearchParams P, const ScreenBufs B) {
  __shared__ unsigned s_h[256], s_bits, s_left;
  const unsigned n = min(B.n[0], B.pilot_cap);
  const unsigned K = (unsigned)P.top_k;
  unsigned thr = 0x7F800000u;  // +inf
  if (n >= K) {
    unsigned bits = 0, mask = 0;
    if (threadIdx.x == 0) s_left = K;
    for (int sh = 24; sh >= 0; sh -= 8) {
      s_h[threadIdx.x] = 0;
      __syncthreads();
      for (unsigned i = threadIdx.x; i < n; i += 256) {
        const unsigned b = __float_as_uint(B.ub[i]);
        if ((b & mask) == bits) atomicAdd(&s_h[(b >> sh) & 255u], 1u);
      }
      __syncthreads();
      if (threadIdx.x < 32) {  // the bin that holds the s_left-th
        unsigned h[8], t = 0;
        for (int k = 0; k < 8; ++k) {
          h[k] = s_h[threadIdx.x * 8 + k];
          t += h[k];
        }
        unsigned p = t;
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned v = __shfl_up_sync(kFull, p, o);
          if (threadIdx.x >= o) p += v;
        }
        unsigned below = p - t;
        const unsigned left = s_left;
        __syncwarp();
        if (below < left && p >= left) {
          for (int k = 0; k < 8; ++k) {
            if (below + h[k] >= left) {
              s_bits = bits | ((threadIdx.x * 8 + k) << sh);
              s_left = left - below;
              break;
            }
            below += h[k];
          }
        }
      }
      __syncthreads();
      bits = s_bits;
      mask |= 255u << sh;
    }
    thr = bits;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && thr < 0x7F800000u)
    atomicMin(P.gthr, (unsigned long long)__double_as_longlong(
                          (double)__uint_as_float(thr)));
  // a code is the upper half of its bound's bits: bound <= thr needs
  // code <= thr >> 16
  const unsigned cut = thr >> 16;
  append(B, (unsigned)P.count, B.list_cap, B.list, &B.n[1],
         [=](unsigned code, unsigned) { return code <= cut; });
}

}  // namespace

cudaError_t launch_screen(const SearchParams &P, const ScreenBufs &B,
                          int sm_count, cudaStream_t st) {
  const long long tiles = (P.count + 63) / 64;
  const long long want = (tiles + kScreenThreads / 32 - 1) /
                         (kScreenThreads / 32);
  const int grid = (int)std::min<long long>(want, 4LL * sm_count);
  if (P.quadh)
    k_screen<true><<<grid, kScreenThreads, 0, st>>>(P, B);
  else
    k_screen<false><<<grid, kScreenThreads, 0, st>>>(P, B);
  return cudaGetLastError();
}

static int append_grid(const SearchParams &P, int sm_count) {
  const long long want = (P.count + 2047) / 2048;
  return (int)std::min<long long>(want, 2LL * sm_count);
}

cudaError_t launch_screen_pilot_list(const SearchParams &P,
                                     const ScreenBufs &B, int sm_count,
                                     cudaStream_t st) {
  k_pilot_list<<<append_grid(P, sm_count), 256, 0, st>>>(P, B);
  return cudaGetLastError();
}

cudaError_t launch_screen_pilot(const SearchParams &P, const ScreenBufs &B,
                                size_t smem_optin, int sm_count,
                                cudaStream_t st) {
  const int per = kPilotTpg * kPilotWarps;
  const int grid = (int)((B.pilot_cap + per - 1) / per);
  const size_t sm = sizeof(float4) * (size_t)P.n_ep;
  (void)sm_count;
  (void)smem_optin;
  // staged while two blocks fit an SM
  if (sm <= 100 * 1024) {
    static int set_of[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64 || !set_of[dev]) {
      cudaFuncSetAttribute(k_pilot<true, true>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           100 * 1024);
      cudaFuncSetAttribute(k_pilot<true, false>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           100 * 1024);
      if (dev < 64) set_of[dev] = 1;
    }
    if (P.quadh)
      k_pilot<true, true><<<grid, kPilotWarps * 32, sm, st>>>(P, B);
    else
      k_pilot<true, false><<<grid, kPilotWarps * 32, sm, st>>>(P, B);
  } else if (P.quadh) {
    k_pilot<false, true><<<grid, kPilotWarps * 32, 0, st>>>(P, B);
  } else {
    k_pilot<false, false><<<grid, kPilotWarps * 32, 0, st>>>(P, B);
  }
  return cudaGetLastError();
}

cudaError_t launch_screen_list(const SearchParams &P, const ScreenBufs &B,
                               int sm_count, cudaStream_t st) {
  k_list<<<append_grid(P, sm_count), 256, 0, st>>>(P, B);
  return cudaGetLastError();
}

}  // namespace morse
