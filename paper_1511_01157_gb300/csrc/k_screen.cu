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
//   k_pilot        upper bounds of their chi^2 over the whole light curve,
//                  and the third subset's bounds of a sample of the grid
//   k_list         the K-th of those, a rigorous threshold near the final
//                  one, and the list of trajectories at or below it; or no
//                  list, where the sample says that it would be too long
//   k_rescreen     the listed ones again, on the second and third subsets
//
// The listed search (k_search_list) then runs over the list alone, with the
// largest subset first.  Results are those of the unscreened search bit for
// bit: a discarded trajectory's chi^2 exceeds K others', and every listed
// one is evaluated by the same device functions.  Measured, call by call
// (1024^2 map, 1.44 M trajectories, 3000 epochs, K = 256, five events of
// tE 7 to 37 d): 3.2 -> 0.45 to 1.3 ms, four maps of a sweep 13 -> 2.0 to
// 4.5 ms; the spread is the light curves' own (what share of the grid fits
// them about as well as the best).  The host screens from 16 384
// trajectories and 128 epochs on; below that a search is bound by its
// launches and its latency, and there are too few trajectories to rank.
// Where the subsets discard too little the whole range is searched as before
// (k_search).  Light curves whose signal is too weak for them are known on the
// host and not screened (screen_subsets); the others cost the first subset's
// walk (32 of up to 639 epochs, 64 of more: a share of 25 % at 128 epochs, 16
// at 200, 2 at 3000, less what the pilot's threshold saves) and five launches
// before a sample shows it: up to 5 % of a search of 300 000 trajectories,
// 18 % in the worst case seen (k_list).
//
// Grids of up to kSmallGrid trajectories are too few to rank by subsets and
// bound by latency: k_bounds takes upper and lower bounds of all of them over
// the whole light curve, spread over every SM (in k_search they are the FP64
// solves and the ordered merges of 16 warps on a few SMs), and k_list and the
// listed search follow.  3600 trajectories x 201 epochs, a call: 208 -> 111
// us.
#ifndef MORSE_PK_ASM
#define MORSE_PK_ASM 1
#endif
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "morse_internal.cuh"
#include "search_common.cuh"

namespace morse {

namespace {

using namespace dev;

constexpr int kScreenThreads = 256;
constexpr int kScreenTile = 2 * kScreenThreads;  // trajectories per block step
// epochs of the subsets, at most
constexpr int kScreenMax0 = 128, kScreenMax1 = 192, kScreenMax2 = 1024;

// Order of the trajectories in a screen.  The grid index runs over tE
// fastest; here the position in a line runs over t0 fastest, so that the
// lanes of a warp, at the same epoch, sit at neighbouring places of the
// line and their 16-byte cells share cache lines (tE is log-spaced: at the
// same t0 its values spread over the whole line).  A range that does not
// consist of whole lines keeps the grid order.
struct Pos {
  unsigned line, it0, itE;
};
__device__ __forceinline__ bool by_t0(const SearchParams &P) {
  return P.first % P.line == 0 && P.count % P.line == 0;
}
__device__ __forceinline__ Pos pos_of(const SearchParams &P, unsigned p,
                                      bool t0_fast) {
  const unsigned n = (unsigned)P.line;
  Pos o;
  if (t0_fast) {
    o.line = p / n;
    const unsigned r = p - o.line * n;
    o.itE = r / (unsigned)P.n_t0;
    o.it0 = r - o.itE * (unsigned)P.n_t0;
    o.line += (unsigned)(P.first / P.line);
  } else {
    const unsigned j = (unsigned)P.first + p;
    o.line = j / n;
    const unsigned r = j - o.line * n;
    o.it0 = r / (unsigned)P.n_tE;
    o.itE = r - o.it0 * (unsigned)P.n_tE;
  }
  return o;
}
// offset of a position's trajectory from P.first
__device__ __forceinline__ unsigned offset_of(const SearchParams &P,
                                              unsigned p, bool t0_fast) {
  if (!t0_fast) return p;
  const unsigned n = (unsigned)P.line, l = p / n, r = p - l * n;
  const unsigned itE = r / (unsigned)P.n_t0;
  return l * n + (r - itE * (unsigned)P.n_t0) * (unsigned)P.n_tE + itE;
}

// The FP64 constants that the trajectories of one (line, tE) share (a row:
// n_t0 positions), made once per row of a block's tile: an FP64 instruction
// holds the SM's FP64 pipe for some 16 cycles, and 15 of a trajectory's 26
// do not depend on its t0.
struct Row {
  double ax, ay, cx, cy, kt, tE, tlo, thi, lsh;
  float axf, ayf, ktf, u02;
};
constexpr int kRowMax = 176;  // rows of a tile: kScreenTile / n_t0 + 2

__device__ __forceinline__ Row make_row(const SearchParams &P, unsigned line,
                                        unsigned itE) {
  // (the operations of traj_base_of and traj_base, in their order)
  const unsigned iu = line / (unsigned)P.n_alpha;
  const unsigned ia = line - iu * (unsigned)P.n_alpha;
  const double2 sl = P.slab[line];
  double u, c, s, k = P.invtEd[itE];
  Row r;
  r.tE = P.tEv[itE];
  r.lsh = 0.0;
  if (P.lu) {
    if (P.ltE) {
      r.tE = P.ltE[iu];
      k = 1.0 / (r.tE * P.dlt);
    }
    r.lsh = P.lsh[iu];
    u = P.lu[iu];
    c = P.lc[iu];
    s = P.ls[iu];
  } else {
    u = P.u0v[iu];
    c = P.ca[ia];
    s = P.sa[ia];
  }
  r.ax = __dmul_rn(c, k);
  r.ay = __dmul_rn(s, k);
  r.cx = __dadd_rn(__dmul_rn(-__dmul_rn(u, s), P.invD), P.coff);
  r.cy = __dadd_rn(__dmul_rn(__dmul_rn(u, c), P.invD), P.coff);
  r.kt = __dmul_rn(k, P.dlt);
  r.tlo = sl.x;
  r.thi = sl.y;
  r.axf = __double2float_rn(r.ax);
  r.ayf = __double2float_rn(r.ay);
  r.ktf = __double2float_rn(r.kt);
  r.u02 = __double2float_rn(__dmul_rn(u, u));
  return r;
}

// a trajectory of a row: its constants and the FP32 times between which it
// is inside the map (in < t < out)
__device__ __forceinline__ TrajC row_traj(const SearchParams &P, const Row &r,
                                          unsigned it0, float &in,
                                          float &out) {
  double t0 = P.t0rel[it0];
  if (P.lu) t0 = t0 - r.lsh * r.tE;
  TrajC o;
  o.ax = r.axf;
  o.ay = r.ayf;
  o.bx = __double2float_rn(__dsub_rn(r.cx, __dmul_rn(t0, r.ax)));
  o.by = __double2float_rn(__dsub_rn(r.cy, __dmul_rn(t0, r.ay)));
  o.kt = r.ktf;
  o.bt = __double2float_rn(-__dmul_rn(t0, r.kt));
  o.u02 = r.u02;
  if (r.tlo < r.thi) {
    in = __double2float_rd(t0 + r.tlo * r.tE);
    out = __double2float_ru(t0 + r.thi * r.tE);
  } else {
    in = out = CUDART_INF_F;
  }
  o.e_in = o.e_out = 0;
  return o;
}

// The cells a lane looked up last.  The subsets are runs of neighbouring
// epochs, so a trajectory mostly stays in its cell from one epoch to the
// next, and only the lanes that leave theirs load another: a warp's gather
// of 32 cells takes 12 wavefronts of the L1 data pipe, which bounded the
// screen (157 us of 1.44 M trajectories x 64 epochs).
template <bool H>
struct Cells {
  unsigned ia, ib;
  float4 a, b;  // FP32 cells; FP16: decoded (band_cell_h)
};

template <bool H>
__device__ __forceinline__ float4 load_cell(const SearchParams &P,
                                            unsigned idx) {
  return H ? band_cell_h(__ldg(&P.quadh[idx])) : __ldg(&P.quad[idx]);
}

// A - 1 of both inside the map (the arithmetic of tex_pos and bilinear_m1 or
// bilinear_h_m1, the coordinates packed)
template <bool H>
__device__ __forceinline__ float2 in2_m1(const SearchParams &P, Cells<H> &q,
                                         float2 vx, float2 vy) {
  float2 fx, fy;
  unsigned ia, ib;
  TexPos ta, tb;
  if (!tex_pos(P, vx.x, vy.x, ta) || !tex_pos(P, vx.y, vy.y, tb))
    return make_float2(0.f, 0.f);  // (checked build only)
  if (kTileW == 1 && kTileH == 1) {
    const float2 tx = pk_add_rd(vx, f2(12582912.f));
    const float2 ty = pk_add_rd(vy, f2(12582912.f));
    fx = pk_fma(pk_add(tx, f2(-12582912.f)), f2(-1.f), vx);
    fy = pk_fma(pk_add(ty, f2(-12582912.f)), f2(-1.f), vy);
    const unsigned qp = (unsigned)P.qpitch;
    ia = __float_as_uint(ty.x) * qp + __float_as_uint(tx.x) + P.qidx0;
    ib = __float_as_uint(ty.y) * qp + __float_as_uint(tx.y) + P.qidx0;
  } else {
    fx = make_float2(ta.fx, tb.fx);
    fy = make_float2(ta.fy, tb.fy);
    ia = ta.idx;
    ib = tb.idx;
  }
  const bool na = ia != q.ia, nb = ib != q.ib;
  q.ia = ia;
  q.ib = ib;
  if (na) q.a = load_cell<H>(P, ia);
  if (nb) q.b = load_cell<H>(P, ib);
  const float2 r0 = pk_fma(fx, make_float2(q.a.y, q.b.y),
                           make_float2(q.a.x, q.b.x));
  const float2 dr = pk_fma(fx, make_float2(q.a.w, q.b.w),
                           make_float2(q.a.z, q.b.z));
  const float2 v = pk_fma(fy, dr, r0);
  return H ? make_float2(__fsub_rn(v.x, 1.f), __fsub_rn(v.y, 1.f)) : v;
}

// The subset's bounds for two trajectories of a lane (packed FP32), every
// lane over the whole subset: no reductions, one broadcast shared load of
// an epoch for the warp's 64 trajectories.  Or, with lg > 0, 2^lg neighbouring
// lanes have the same two trajectories, each an equal piece of the subset
// (split_len; the last past its end: pad_subset), and the sums are
// added across them (the bound's error covers any order).
constexpr int kSplitMax = 2;   // 4 lanes a trajectory at most
constexpr int kSplitPad = 8;   // epochs past the subset: 2 x lanes - 1, or less
__device__ __forceinline__ int split_len(int m, int lg) {
  // odd: the lanes' pieces start in different banks
  return lg ? ((m + (1 << lg) - 1) >> lg) | 1 : m;
}
template <bool H>
__device__ __forceinline__ void screen2(const SearchParams &P,
                                        const ScreenLv &V, const float4 *s_ep,
                                        const TrajC &ca, const TrajC &cb,
                                        float ain, float aout, float bin,
                                        float bout, float &la, float &lb,
                                        int lg = 0) {
  const TrajP c = pack_traj(ca, cb);
  const float hi = fmaxf(ain, bin), lo = fminf(aout, bout);
  Acc2 s = {f2(0.f), f2(0.f), f2(0.f)};
  Cells<H> q;
  q.ia = q.ib = 0xFFFFFFFFu;
  q.a = q.b = make_float4(0.f, 0.f, 0.f, 0.f);
  const int len = split_len(V.m, lg);
  s_ep += ((int)threadIdx.x & ((1 << lg) - 1)) * len;
#pragma unroll 4
  for (int e = 0; e < len; ++e) {
    const float4 v = s_ep[e];
    const float2 tt = f2(v.x);
    const float2 vx = pk_fma(c.ax, tt, c.bx);
    const float2 vy = pk_fma(c.ay, tt, c.by);
    float2 Ac;
    if (__all_sync(kFull, v.x > hi && v.x < lo)) {  // all of the warp inside
      Ac = in2_m1<H>(P, q, vx, vy);
    } else {
      const bool ina = v.x > ain && v.x < aout;
      const bool inb = v.x > bin && v.x < bout;
      Ac = mag2_out_m1(c, tt);
      if (__any_sync(kFull, ina || inb)) {
        // (outside: a cell of the map's centre, the value is not used)
        const float2 A =
            in2_m1<H>(P, q, make_float2(ina ? vx.x : 0.f, inb ? vx.y : 0.f),
                      make_float2(ina ? vy.x : 0.f, inb ? vy.y : 0.f));
        if (ina) Ac.x = A.x;
        if (inb) Ac.y = A.y;
      }
    }
    acc2_add(s, f2(v.y), f2(v.z), Ac);
  }
  for (int o = 1; o < 1 << lg; o <<= 1) {
    s.a = pk_add(s.a, make_float2(__shfl_xor_sync(kFull, s.a.x, o),
                                  __shfl_xor_sync(kFull, s.a.y, o)));
    s.b = pk_add(s.b, make_float2(__shfl_xor_sync(kFull, s.b.x, o),
                                  __shfl_xor_sync(kFull, s.b.y, o)));
    s.d = pk_add(s.d, make_float2(__shfl_xor_sync(kFull, s.d.x, o),
                                  __shfl_xor_sync(kFull, s.d.y, o)));
  }
  const Acc sa = {s.a.x, s.b.x, s.d.x}, sb = {s.a.y, s.b.y, s.d.y};
  la = screen_lb(V, sa);
  lb = screen_lb(V, sb);
}

__device__ __forceinline__ void stage_subset(const ScreenLv &V,
                                             float4 *s_ep) {
  const Epochs ep = epochs_at(V.ep, V.m);
  for (int e = threadIdx.x; e < V.m; e += blockDim.x)
    s_ep[e] = make_float4(ep.tw[e].x, ep.tw[e].y, ep.wf[e], 0.f);
}
// epochs without weight after the subset's (for the lanes of split_len)
__device__ __forceinline__ void pad_subset(const ScreenLv &V, float4 *s_ep) {
  const float t = epochs_at(V.ep, V.m).tw[V.m - 1].x;
  for (int e = threadIdx.x; e < kSplitPad; e += blockDim.x)
    s_ep[V.m + e] = make_float4(t, 0.f, 0.f, 0.f);
}

// Codes of all trajectories, on the smallest subset.
template <bool H>
__device__ __forceinline__ void screen_all(const SearchParams &P,
                                           const ScreenBufs &B) {
  __shared__ float4 s_ep[kScreenMax0];
  __shared__ unsigned s_hist[kScreenBins];
  __shared__ Row s_row[kRowMax];
  const ScreenLv V = P.lv[0];
  stage_subset(V, s_ep);
  for (int b = threadIdx.x; b < kScreenBins; b += blockDim.x) s_hist[b] = 0;
  const bool tf = by_t0(P);
  const unsigned n = (unsigned)P.count, n_t0 = (unsigned)P.n_t0;
  const bool rows = tf && n_t0 >= 3;
  const unsigned row_first = rows ? (unsigned)(P.first / n_t0) : 0u;
  for (unsigned c0 = blockIdx.x * kScreenTile; c0 < n;
       c0 += gridDim.x * kScreenTile) {
    __syncthreads();  // the subset, the histogram; the last tile's rows read
    const unsigned r0 = c0 / n_t0;
    if (rows) {
      const unsigned r1 = (min(c0 + kScreenTile, n) - 1) / n_t0;
      for (unsigned r = r0 + threadIdx.x; r <= r1; r += blockDim.x) {
        const unsigned row = row_first + r;
        const unsigned line = row / (unsigned)P.n_tE;
        s_row[r - r0] = make_row(P, line, row - line * (unsigned)P.n_tE);
      }
      __syncthreads();
    }
    const unsigned pa = c0 + (threadIdx.x >> 5) * 64 + (threadIdx.x & 31);
    const unsigned pb = pa + 32;
    TrajC c[2];
    float in[2], out[2];
    bool cut[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned p = min(h ? pb : pa, n - 1);
      unsigned line;
      if (rows) {
        const unsigned r = p / n_t0;
        c[h] = row_traj(P, s_row[r - r0], p - r * n_t0, in[h], out[h]);
        line = (row_first + r) / (unsigned)P.n_tE;
      } else {
        const Pos o = pos_of(P, p, tf);
        c[h] = row_traj(P, make_row(P, o.line, o.itE), o.it0, in[h], out[h]);
        line = o.line;
      }
      // trajectories of cut lines are not searched
      cut[h] = P.linemax && __ldg(&P.linemax[line]) < P.a_min;
    }
    float la = 0.f, lb = 0.f;
    if (__any_sync(kFull, !cut[0] || !cut[1]))
      screen2<H>(P, V, s_ep, c[0], c[1], in[0], out[0], in[1], out[1], la,
                 lb);
    const unsigned ka = cut[0] ? kScreenCut : __float_as_uint(la) >> 16;
    const unsigned kb = cut[1] ? kScreenCut : __float_as_uint(lb) >> 16;
    if (pa < n) {
      B.code[pa] = (unsigned short)ka;
      if (!cut[0]) atomicAdd(&s_hist[ka / kScreenBinCodes], 1u);
    }
    if (pb < n) {
      B.code[pb] = (unsigned short)kb;
      if (!cut[1]) atomicAdd(&s_hist[kb / kScreenBinCodes], 1u);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kScreenBins; b += blockDim.x)
    if (s_hist[b]) atomicAdd(&B.hist[b], s_hist[b]);
}

constexpr int kListThreads = 1024;  // blocks of the two list kernels

// Appends the trajectories keep() accepts to out[], in ascending order
// within a block's chunks of codes (one atomic per chunk): neighbouring
// entries mostly share a line of the map.
template <typename Keep>
__device__ __forceinline__ void append(const SearchParams &P,
                                       const ScreenBufs &B, unsigned cap,
                                       unsigned *out, unsigned *len,
                                       const Keep &keep) {
  constexpr int kPer = 8;  // codes per thread: one 16-byte load
  const unsigned n = (unsigned)P.count;
  const bool tf = B.pilot && by_t0(P);  // (small grids: the grid order)
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
    if (warp == 0) {
      const unsigned v = lane < nw ? s_w[lane] : 0u;
      unsigned t = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(kFull, t, o);
        if (lane >= o) t += u;
      }
      if (lane < nw) s_w[lane] = t - v;
      if (lane == 31) s_base = t ? atomicAdd(len, t) : 0u;
    }
    __syncthreads();
    unsigned at = s_base + s_w[warp] + p - c;
    for (; m; m &= m - 1, ++at)
      if (at < cap) out[at] = offset_of(P, i0 + (__ffs(m) - 1), tf);
    __syncthreads();
  }
}

// The pilot's list: every trajectory below the histogram bin that holds the
// want-th lowest code, and a hashed sample of that bin's (codes are equal
// there as far as the histogram tells: all of them, where the bounds say
// nothing).
__device__ __forceinline__ void make_pilot_list(const SearchParams &P,
                                                const ScreenBufs &B) {
  __shared__ unsigned s_w[32], s_cut, s_r;
  static_assert(kScreenBins == kListThreads, "a bin per thread");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned h = B.hist[threadIdx.x];
  unsigned p = h;  // cumulated
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(kFull, p, o);
    if (lane >= o) p += v;
  }
  if (lane == 31) s_w[warp] = p;
  if (threadIdx.x == 0) {
    s_cut = kScreenBins;
    s_r = 1;
  }
  __syncthreads();
  for (int w = 0; w < warp; ++w) p += s_w[w];
  if (p >= B.want && p - h < B.want) {
    const unsigned left = B.want - (p - h);
    s_cut = threadIdx.x;
    s_r = (h + left - 1) / left;
  }
  __syncthreads();
  const unsigned cut = s_cut, r = s_r;
  append(P, B, B.pilot_cap, B.pilot, &B.n[0],
         [=](unsigned code, unsigned i) {
           const unsigned b = code / kScreenBinCodes;
           return b < cut ||
                  (b == cut && ((i * 0x9E3779B1u) >> 8) % r == 0u);
         });
}

// Upper bounds of the pilot's chi^2 over the whole light curve (chi2_upper).
// A block takes kPilotTpg entries, its warps a slice of the epochs each (a
// few thousand entries would leave most of the chip waiting for the walk of
// one warp), and one warp adds the slices and solves.
constexpr int kPilotTpg = 8, kPilotWarps = 8;

// The third subset's bounds of kScreenSample trajectories spread over the
// grid, a warp each, in blocks of their own after the pilot's: what part of
// the grid the rescreening would discard, before it is begun (make_list).
// (-1: on a cut line.)
constexpr int kSampleBlocks = kScreenSample / kPilotWarps;
template <bool H>
__device__ __forceinline__ void sample_bounds(const SearchParams &P,
                                              const ScreenBufs &B,
                                              unsigned block) {
  if (P.n_lv < 3) return;
  const int lane = threadIdx.x & 31;
  const unsigned s = block * kPilotWarps + (threadIdx.x >> 5);
  const ScreenLv &V = P.lv[2];
  // multiples of the golden ratio: no stride of the grid's axes
  const unsigned j =
      (unsigned)P.first + __umulhi(s * 0x9E3779B1u, (unsigned)P.count);
  double xi, xo;
  TrajC c = traj_base_of(P, j, xi, xo);
  const Epochs ep = epochs_at(V.ep, V.m);
  traj_range(ep, V.m, xi, xo, c);
  Acc a, b;
  phase1_pair_n<H>(P, ep, V.m, c, c, lane, a, b);
  const bool cut =
      P.linemax && __ldg(&P.linemax[j / (unsigned)P.line]) < P.a_min;
  if (lane == 0) B.smp[s] = cut ? -1.f : screen_lb(V, a);
}

// ALL: the entries are the trajectories themselves (small grids), and their
// lower bounds (solve2's) are coded too.
template <bool H, bool ALL>
__device__ __forceinline__ void pilot_bounds(const SearchParams &P,
                                             const ScreenBufs &B) {
  __shared__ Acc s_acc[kPilotWarps][kPilotTpg];
  __shared__ TrajC s_c[kPilotTpg];
  if (!ALL) {
    const unsigned pilots = gridDim.x - kSampleBlocks;
    if (blockIdx.x >= pilots) {
      sample_bounds<H>(P, B, blockIdx.x - pilots);
      return;
    }
  }
  const unsigned n = ALL ? (unsigned)P.count : min(B.n[0], B.pilot_cap);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned g0 = blockIdx.x * kPilotTpg;
  if (g0 >= n) return;
  const int nv = (int)min((unsigned)kPilotTpg, n - g0);
  Epochs ep = epochs_at(P.ep, P.n_ep);
  if (warp == 0) {  // once: the constants' FP64 would be the block's limit
    double xi, xo;
    const unsigned k = g0 + (lane < nv ? lane : 0);
    TrajC c = traj_base_of(P, (unsigned)P.first + (ALL ? k : B.pilot[k]), xi,
                           xo);
    traj_range(ep, P.n_ep, xi, xo, c);
    if (lane < kPilotTpg) s_c[lane] = c;
  }
  __syncthreads();
  TrajC mine = s_c[lane < kPilotTpg ? lane : 0];
  const int e0 = (int)((long long)P.n_ep * warp / kPilotWarps);
  const int m = (int)((long long)P.n_ep * (warp + 1) / kPilotWarps) - e0;
  ep.tw += e0;
  ep.wf += e0;
  mine.e_in = min(max(mine.e_in - e0, 0), m);
  mine.e_out = min(max(mine.e_out - e0, 0), m);
  for (int k = 0; k < nv; k += 2) {
    const int k2 = min(k + 1, nv - 1);
    const TrajC ca = shfl_traj(mine, k), cb = shfl_traj(mine, k2);
    Acc ra, rb;
    phase1_pair_n<H>(P, ep, m, ca, cb, lane, ra, rb);
    if (lane == 0) {
      s_acc[warp][k] = ra;
      s_acc[warp][k2] = rb;
    }
  }
  __syncthreads();
  if (warp != 0) return;
  Acc ms = {0.f, 0.f, 0.f};
  if (lane < nv)
    for (int w = 0; w < kPilotWarps; ++w) {
      ms.a += s_acc[w][lane].a;
      ms.b += s_acc[w][lane].b;
      ms.d += s_acc[w][lane].d;
    }
  const Fit2 f = fit2(P, (double)ms.a, (double)ms.b, (double)ms.d);
  // the relative error of the slices' sums, as event_params bounds a whole
  // one's: the terms of a lane, the butterfly and the slices
  const float terms =
      (float)(P.n_ep / kPilotWarps / 32 + 2 + 10 + kPilotWarps);
  const double gamma = fmax(P.gamma, (double)(terms * 5.9604645e-8f));
  const double ub =
      chi2_upper(P, (double)ms.a, (double)ms.b, (double)ms.d,
                 (double)__double2float_rn(f.Fs),
                 (double)__double2float_rn(f.Bc), gamma);
  float up = fmaxf(__double2float_ru(ub), 0.f);
  if (ALL) {
    SearchParams Q = P;
    Q.gamma = gamma;
    const Solved o =
        solve2(Q, (double)ms.a, (double)ms.b, (double)ms.d);
    // may_reach's bound and margin, rounded down
    const double lb =
        o.bden > 0.0 ? (P.CFF - o.bnum / o.bden) * (1.0 - 1.01e-4) : 0.0;
    unsigned code = __float_as_uint(lb > 0.0 ? __double2float_rd(lb) : 0.f)
                    >> 16;
    if (P.linemax && lane < nv &&
        __ldg(&P.linemax[((unsigned)P.first + g0 + lane) /
                         (unsigned)P.line]) < P.a_min) {
      code = kScreenCut;  // not searched, and no bound for the others
      up = CUDART_INF_F;
    }
    if (lane < nv) B.code[g0 + lane] = (unsigned short)code;
  }
  if (lane < nv) B.ub[g0 + lane] = up;
}

// The sample has to discard one in kSampleGive.  Small-u0 shares of a grid
// (ranges of it), whose trajectories all miss the light curve by about as
// much, and variables that none fits, 60 000 and 300 000 trajectories, 1100
// to 8000 epochs: 1.10 to 1.55 times the unscreened search without the rule,
// 0.91 to 1.06 with it (1.18 for the variable of 1100 epochs and 300 000).
// One in 2 and one in 3 did the same there, but a batch whose lists leave out
// a quarter took up to 15 % more.  256 samples know the share to 2 %.
constexpr int kSampleGive = 8;

// The threshold: the top_k-th smallest of the pilot's bounds (K distinct
// trajectories have chi^2 at or below it), by four passes of eight bits
// over the FP32 bit patterns, every block for itself; then the list.
__device__ __forceinline__ void make_list(const SearchParams &P,
                                          const ScreenBufs &B) {
  __shared__ unsigned s_h[256], s_bits, s_left;
  const unsigned n =
      B.pilot ? min(B.n[0], B.pilot_cap) : (unsigned)P.count;
  const unsigned K = (unsigned)P.top_k;
  unsigned thr = 0x7F800000u;  // +inf
  if (n >= K) {
    unsigned bits = 0, mask = 0;
    if (threadIdx.x == 0) s_left = K;
    for (int sh = 24; sh >= 0; sh -= 8) {
      if (threadIdx.x < 256) s_h[threadIdx.x] = 0;
      __syncthreads();
      for (unsigned i = threadIdx.x; i < n; i += kListThreads) {
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
  // No list when the sample's bounds discard too few (a light curve that no
  // trajectory of the range fits, whose threshold no subset's chi^2 reaches).
  if (P.n_lv > 2) {
    static_assert(kScreenSample <= kListThreads, "a sample per thread");
    const float lb =
        threadIdx.x < kScreenSample ? B.smp[threadIdx.x] : -1.f;
    const int all = __syncthreads_count(lb >= 0.f);
    const int gone = __syncthreads_count(lb > __uint_as_float(thr));
    if (kSampleGive * gone < all) {  // (the same in every block)
      if (blockIdx.x == 0 && threadIdx.x == 0) B.n[4] = 1u;
      return;
    }
  }
  // a code is the upper half of its bound's bits: bound <= thr needs
  // code <= thr >> 16
  const unsigned cut = thr >> 16;
  append(P, B, B.list0_cap, B.list0, &B.n[1],
         [=](unsigned code, unsigned) { return code <= cut; });
}

// The listed trajectories on the second and third subsets, now against the
// threshold: those left go to the final list.  A block keeps what the second
// subset leaves in a queue and takes the third with full warps.  When the
// two discard less than one in eight of those decided so far (from 16 384
// on), the screen gives up and the whole range is searched.
//
// A short list leaves SMs without a tile, and a lane's walk over the subset
// is a chain of cell loads: the lanes of a tile then take fewer trajectories,
// 2 or 4 lanes each, while every tile still has a block of its own.  Not in a
// batch, whose other pairs fill the SMs.  Peak-aligned searches (345 600
// trajectories) 621, 616, 615, 690 -> 591, 556, 548, 634 us, a grid of 1.44 M
// whose list is short 452 -> 393, the others within 1.5 %; with 8 lanes the
// same, and the final list's order (tile by tile) gets worse for its search.
template <bool H>
__device__ __forceinline__ void rescreen_listed(const SearchParams &P,
                                                const ScreenBufs &B) {
  if (P.n_lv < 3) return;  // (of a batch: the list is final)
  __shared__ float4 s_e1[kScreenMax1 + kSplitPad],
      s_e2[kScreenMax2 + kSplitPad];
  __shared__ unsigned s_queue[2 * kScreenTile];
  __shared__ unsigned s_m[kScreenThreads / 16], s_base, s_stop;
  const ScreenLv V1 = P.lv[1], V2 = P.lv[2];
  const unsigned n = B.n[1];
  int lg = 0;
  if (gridDim.y == 1)
    while (lg < kSplitMax && ((unsigned long long)n << (lg + 1)) <=
                                 (unsigned long long)gridDim.x * kScreenTile)
      ++lg;
  const unsigned tile = (unsigned)kScreenTile >> lg;
  unsigned c0 = blockIdx.x * tile;
  if (c0 >= n) return;
  stage_subset(V1, s_e1);
  stage_subset(V2, s_e2);
  pad_subset(V1, s_e1);
  pad_subset(V2, s_e2);
  const float thr = __double2float_ru(bits_to_chi2(__ldcg(P.gthr)));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  unsigned queued = 0;  // block-uniform
  while (c0 < n || queued > 0) {
    const bool first = c0 < n && queued < tile;
    const unsigned m = min(tile, first ? n - c0 : queued);
    const unsigned q0 = first ? 0u : queued - m;
    if (threadIdx.x == 0) s_stop = *(volatile unsigned *)&B.n[4];
    __syncthreads();  // the subsets, the queue
    if (s_stop) return;
    const unsigned w0 = ((unsigned)warp * 64u) >> lg;
    const unsigned i[2] = {w0 + ((unsigned)lane >> lg),
                           w0 + ((unsigned)(lane + 32) >> lg)};
    const bool lead = (lane & ((1 << lg) - 1)) == 0;  // of a trajectory
    unsigned off[2];
    TrajC c[2];
    float in[2], out[2];
    unsigned ma = 0, mb = 0;
    if (w0 < m) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned k = min(i[h], m - 1);
        off[h] = first ? B.list0[c0 + k] : s_queue[q0 + k];
        double xi, xo;
        c[h] = traj_base_of(P, (unsigned)P.first + off[h], xi, xo);
        in[h] = __double2float_rd(xi);
        out[h] = __double2float_ru(xo);
      }
      float la, lb;
      if (first)
        screen2<H>(P, V1, s_e1, c[0], c[1], in[0], out[0], in[1],
                   out[1], la, lb, lg);
      else
        screen2<H>(P, V2, s_e2, c[0], c[1], in[0], out[0], in[1],
                   out[1], la, lb, lg);
      ma = __ballot_sync(kFull, lead && i[0] < m && la <= thr);
      mb = __ballot_sync(kFull, lead && i[1] < m && lb <= thr);
    }
    if (lane == 0) {
      s_m[2 * warp] = __popc(ma);
      s_m[2 * warp + 1] = __popc(mb);
    }
    __syncthreads();  // also: the queue is read
    if (threadIdx.x == 0) {
      unsigned t = 0;
      for (int k = 0; k < kScreenThreads / 16; ++k) {
        const unsigned v = s_m[k];
        s_m[k] = t;
        t += v;
      }
      s_base = first ? t : (t ? atomicAdd(&B.n[2], t) : 0u);
      const unsigned killed = m - t, done = first ? killed : m;
      const unsigned all = atomicAdd(&B.n[3], done) + done;
      const unsigned gone = atomicAdd(&B.n[5], killed) + killed;
      if (all >= 16384u && 8ull * gone < all) atomicExch(&B.n[4], 1u);
    }
    __syncthreads();
    const unsigned ra = s_m[2 * warp] + __popc(ma & below);
    const unsigned rb = s_m[2 * warp + 1] + __popc(mb & below);
    if (first) {
      if (ma >> lane & 1u) s_queue[queued + ra] = off[0];
      if (mb >> lane & 1u) s_queue[queued + rb] = off[1];
      queued += s_base;
      c0 += gridDim.x * tile;
    } else {
      const unsigned g = s_base;
      if ((ma >> lane & 1u) && g + ra < B.list_cap) B.list[g + ra] = off[0];
      if ((mb >> lane & 1u) && g + rb < B.list_cap) B.list[g + rb] = off[1];
      queued -= m;
    }
  }
}

// The kernels: one search, its parameters by value, or a batch of them
// (blockIdx.y), each block with its search's parameters in shared memory.
__device__ __forceinline__ void load_task(const ScreenTask *t, ScreenTask &s) {
  const uint4 *src = reinterpret_cast<const uint4 *>(t);
  uint4 *dst = reinterpret_cast<uint4 *>(&s);
  for (int i = threadIdx.x; i < (int)(sizeof(ScreenTask) / 16);
       i += blockDim.x)
    dst[i] = __ldg(src + i);
  __syncthreads();
}
#define MORSE_SCREEN_KERNELS(TEMPLATE, NAME, BODY, THREADS, MIN)             \
  TEMPLATE                                                                   \
  __global__ void __launch_bounds__(THREADS, MIN)                            \
      NAME(const SearchParams P, const ScreenBufs B) {                       \
    BODY(P, B);                                                              \
  }                                                                          \
  TEMPLATE                                                                   \
  __global__ void __launch_bounds__(THREADS, MIN)                            \
      NAME##_batch(const ScreenTask *t) {                                    \
    __shared__ ScreenTask s;                                                 \
    load_task(t + blockIdx.y, s);                                            \
    BODY(s.F.S, s.B);                                                        \
  }
#define MORSE_BY_TABLE template <bool H>
#define MORSE_EITHER_TABLE
MORSE_SCREEN_KERNELS(MORSE_BY_TABLE, k_screen, screen_all<H>, kScreenThreads,
                     4)
MORSE_SCREEN_KERNELS(MORSE_EITHER_TABLE, k_pilot_list, make_pilot_list,
                     kListThreads, 1)
#define MORSE_PILOT(P, B) pilot_bounds<H, false>(P, B)
MORSE_SCREEN_KERNELS(MORSE_BY_TABLE, k_pilot, MORSE_PILOT, kPilotWarps * 32, 4)
#undef MORSE_PILOT
MORSE_SCREEN_KERNELS(MORSE_EITHER_TABLE, k_list, make_list, kListThreads, 1)
MORSE_SCREEN_KERNELS(MORSE_BY_TABLE, k_rescreen, rescreen_listed<H>,
                     kScreenThreads, 4)
#undef MORSE_BY_TABLE
#undef MORSE_EITHER_TABLE
#undef MORSE_SCREEN_KERNELS

template <bool H>
__global__ void __launch_bounds__(kPilotWarps * 32, 4)
    k_bounds(const SearchParams P, const ScreenBufs B) {
  pilot_bounds<H, true>(P, B);
}

}  // namespace

cudaError_t launch_screen(const SearchParams &P, const ScreenBufs &B,
                          int sm_count, cudaStream_t st) {
  const long long want = (P.count + kScreenTile - 1) / kScreenTile;
  const int grid = (int)std::min<long long>(want, 4LL * sm_count);
  if (P.quadh)
    k_screen<true><<<grid, kScreenThreads, 0, st>>>(P, B);
  else
    k_screen<false><<<grid, kScreenThreads, 0, st>>>(P, B);
  return cudaGetLastError();
}

static int append_grid(const SearchParams &P, int sm_count) {
  const long long want =
      (P.count + 8LL * kListThreads - 1) / (8LL * kListThreads);
  return (int)std::min<long long>(want, (long long)sm_count);
}

cudaError_t launch_screen_pilot_list(const SearchParams &P,
                                     const ScreenBufs &B, int sm_count,
                                     cudaStream_t st) {
  k_pilot_list<<<append_grid(P, sm_count), kListThreads, 0, st>>>(P, B);
  return cudaGetLastError();
}

cudaError_t launch_screen_pilot(const SearchParams &P, const ScreenBufs &B,
                                cudaStream_t st) {
  const int grid =
      (int)((B.pilot_cap + kPilotTpg - 1) / kPilotTpg) + kSampleBlocks;
  if (P.quadh)
    k_pilot<true><<<grid, kPilotWarps * 32, 0, st>>>(P, B);
  else
    k_pilot<false><<<grid, kPilotWarps * 32, 0, st>>>(P, B);
  return cudaGetLastError();
}

cudaError_t launch_bounds(const SearchParams &P, const ScreenBufs &B,
                          cudaStream_t st) {
  const int grid = (int)((P.count + kPilotTpg - 1) / kPilotTpg);
  if (P.quadh)
    k_bounds<true><<<grid, kPilotWarps * 32, 0, st>>>(P, B);
  else
    k_bounds<false><<<grid, kPilotWarps * 32, 0, st>>>(P, B);
  return cudaGetLastError();
}

cudaError_t launch_screen_list(const SearchParams &P, const ScreenBufs &B,
                               int sm_count, cudaStream_t st) {
  k_list<<<append_grid(P, sm_count), kListThreads, 0, st>>>(P, B);
  return cudaGetLastError();
}

cudaError_t launch_rescreen(const SearchParams &P, const ScreenBufs &B,
                            int sm_count, cudaStream_t st) {
  const int tile = kScreenTile >> kSplitMax;
  const long long want = (P.count + tile - 1) / tile;
  const int grid = (int)std::min<long long>(want, 4LL * sm_count);
  if (P.quadh)
    k_rescreen<true><<<grid, kScreenThreads, 0, st>>>(P, B);
  else
    k_rescreen<false><<<grid, kScreenThreads, 0, st>>>(P, B);
  return cudaGetLastError();
}

template <bool H>
static cudaError_t screen_batch(const ScreenTask *t, int n,
                                const SearchParams &P0, const ScreenBufs &B0,
                                bool rescreen, cudaStream_t st) {
  const unsigned tiles =
      (unsigned)((P0.count + kScreenTile - 1) / kScreenTile);
  const unsigned chunks =
      (unsigned)((P0.count + 8LL * kListThreads - 1) / (8LL * kListThreads));
  const unsigned y = (unsigned)n;
  const unsigned pilot =
      (B0.pilot_cap + kPilotTpg - 1) / kPilotTpg + kSampleBlocks;
  // a few tiles per block amortise the subset's staging and the histogram
  k_screen_batch<H><<<dim3((tiles + 3) / 4, y), kScreenThreads, 0, st>>>(t);
  k_pilot_list_batch<<<dim3(chunks, y), kListThreads, 0, st>>>(t);
  k_pilot_batch<H><<<dim3(pilot, y), kPilotWarps * 32, 0, st>>>(t);
  k_list_batch<<<dim3(chunks, y), kListThreads, 0, st>>>(t);
  if (rescreen)
    k_rescreen_batch<H><<<dim3((tiles + 7) / 8, y), kScreenThreads, 0, st>>>(
        t);
  return cudaGetLastError();
}

cudaError_t launch_screen_batch(const ScreenTask *t, int n,
                                const SearchParams &P0, const ScreenBufs &B0,
                                bool rescreen, cudaStream_t st) {
  return P0.quadh ? screen_batch<true>(t, n, P0, B0, rescreen, st)
                  : screen_batch<false>(t, n, P0, B0, rescreen, st);
}

}  // namespace morse
