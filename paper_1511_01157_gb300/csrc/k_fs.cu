// Finite-source maps (§4.1: each point-source map convolved with radially
// symmetric, limb-darkened source profiles of fixed radii).
//
// out(i, j) = sum_{dx, dy} W(dx, dy) A(i + dx, j + dy), W the source
// profile integrated over the texels within R of the centre (normalised),
// a texel outside the map taking the Paczynski magnification of its centre
// (the lookup's outside rule).
//
// GB300 design: a block computes a 64 x 16 tile of outputs, four adjacent
// ones per thread.  The 16 input rows the tile needs at kernel row dy, 64 +
// 2R texels wide, sit in a circular buffer in shared memory that takes one
// new row per dy, next to that row's weights;
// a thread then walks the row in aligned 16-byte chunks, so one chunk of
// texels and one of weights feed 16 FMAs (4 taps x 4 outputs).  Each row's
// sum is FP32 (at most 2R + 4 terms) and is added to an FP64 accumulator,
// so the rounding does not grow with the source area.  Rows of zero weight
// beyond the disc are skipped by their half-width.  (This kernel,
// k_fs_conv, takes the small sources and those of over some 700 texels,
// k_fs_fold the others.)
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "morse_internal.cuh"

namespace morse {

namespace {

constexpr int kFsTX = 64, kFsTY = 16, kFsOut = 4;  // outputs per thread
constexpr int kFsThreads = (kFsTX / kFsOut) * kFsTY;

// Paczynski A of the centre of texel (x, y) outside the map, in FP32
// (relative error a few 1e-7; halo texels of a large source are many)
__device__ __forceinline__ float pspl_at(int x, int y, float L, float dlt) {
  const float y1 = __fmaf_rn((float)x + 0.5f, dlt, -L);
  const float y2 = __fmaf_rn((float)y + 0.5f, dlt, -L);
  const float u2 = __fmaf_rn(y1, y1, y2 * y2);
  return (u2 + 2.0f) * rsqrtf(u2 * (u2 + 4.0f));
}

// Staged row layout: column c holds x = x0 - Ra + c, Ra = R rounded up to a
// multiple of 4, so that the four outputs of a thread (x0 + 4 tx + k) and
// the taps of any dx fall in 16-byte chunks; Wd = row width in floats.
__host__ __device__ __forceinline__ int fs_ra(int R) { return (R + 3) & ~3; }
__host__ __device__ __forceinline__ int fs_width(int R) {
  return kFsTX + 2 * fs_ra(R) + 4;
}

__global__ void __launch_bounds__(kFsThreads)
    k_fs_conv(const float *__restrict__ A, int npix, double L, int R,
              const float *__restrict__ W, const int *__restrict__ rowhw,
              float *__restrict__ out) {
  extern __shared__ __align__(16) float fs_smem[];
  const int Ra = fs_ra(R), width = fs_width(R);
  float *s_in = fs_smem;                 // [kFsTY][width]
  float *s_w = s_in + kFsTY * width;     // [2 Ra + 4], zero outside the row
  const int tx = threadIdx.x % (kFsTX / kFsOut);
  const int ty = threadIdx.x / (kFsTX / kFsOut);
  const int x0 = blockIdx.x * kFsTX, y0 = blockIdx.y * kFsTY;
  const float Lf = (float)L, dltf = (float)((2.0 * L) / (double)npix);
  double acc[kFsOut];
#pragma unroll
  for (int k = 0; k < kFsOut; ++k) acc[k] = 0.0;
  // Circular buffer of kFsTY staged input rows: at kernel row dy the tile
  // needs rows y0 + dy + r, r < kFsTY, and input row y lives in slot
  // (y - y0 + R) mod kFsTY, so each step stages one new row.
  auto stage = [&](int y, int slot) {
    float *dst = s_in + slot * width;
    for (int c = threadIdx.x; c < width; c += blockDim.x) {
      const int x = x0 - Ra + c;
      dst[c] = (x >= 0 && x < npix && y >= 0 && y < npix)
                   ? A[(size_t)y * npix + x]
                   : pspl_at(x, y, Lf, dltf);
    }
  };
  for (int r = 0; r < kFsTY - 1; ++r) stage(y0 - R + r, r);
  for (int dy = -R; dy <= R; ++dy) {
    stage(y0 + dy + kFsTY - 1, (dy + R + kFsTY - 1) % kFsTY);
    const int hw = rowhw[dy + R];  // weights nonzero for |dx| <= hw
    if (hw < 0) {                  // block-uniform: nothing to add
      __syncthreads();
      continue;
    }
    // weights of this row at dx + Ra, zero beyond the disc
    for (int t = threadIdx.x; t < 2 * Ra + 4; t += blockDim.x) {
      const int dx = t - Ra;
      s_w[t] = (dx >= -hw && dx <= hw)
                   ? W[(size_t)(dy + R) * (2 * R + 1) + (dx + R)]
                   : 0.f;
    }
    __syncthreads();
    // taps dx = dxa - Ra for dxa in [Ra - hw, Ra + hw], in aligned groups
    // of four: output k needs s_in[4 tx + dxa + k]
    const int a0 = (Ra - hw) & ~3, a1 = Ra + hw;
    const float4 *row4 = reinterpret_cast<const float4 *>(
                             s_in + ((ty + dy + R) % kFsTY) * width) +
                         tx;
    const float4 *w4 = reinterpret_cast<const float4 *>(s_w);
    float rs[kFsOut] = {0.f, 0.f, 0.f, 0.f};
    float4 cur = row4[a0 >> 2];
    for (int dxa = a0; dxa <= a1; dxa += 4) {
      const float4 nxt = row4[(dxa >> 2) + 1];
      const float4 w = w4[dxa >> 2];
      const float v[8] = {cur.x, cur.y, cur.z, cur.w,
                          nxt.x, nxt.y, nxt.z, nxt.w};
      const float ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int k = 0; k < kFsOut; ++k)
          rs[k] = __fmaf_rn(ww[o], v[o + k], rs[k]);
      cur = nxt;
    }
#pragma unroll
    for (int k = 0; k < kFsOut; ++k) acc[k] += (double)rs[k];
    __syncthreads();
  }
  const int y = y0 + ty;
#pragma unroll
  for (int k = 0; k < kFsOut; ++k) {
    const int x = x0 + kFsOut * tx + k;
    if (x < npix && y < npix) out[(size_t)y * npix + x] = (float)acc[k];
  }
}

// The same convolution folded about the source's axis: W(dx, -dy) = W(dx,
// dy), so the input rows y + dy and y - dy are added first, once for all dx,
// and every weight is applied to the sum (of halves, by twice the weight: the
// sum stays in FP32's range with its texels): half the multiply-adds, which
// bound k_fs_conv (with the FP64 additions of its row sums: two FP64-pipe
// instructions per output and row, some 16 cycles each per warp).
//
// A block computes 64 x 16 outputs with G groups of 128 threads, eight
// adjacent outputs per thread; a group takes its share of a row's taps (more
// warps for the same staged rows, which for a large source fill the SM's
// shared memory, and shorter FP32 sums; two groups up to R = 140, four
// beyond: with four a row of R = 77 is five steps per thread, less than its
// staging costs).  The rows sit in two circular
// buffers (rows moving up, rows moving down) with a slot to spare each: the
// next dy's two rows and weights are loaded into registers before the sums
// of dy and stored after them, one barrier per dy.  Two chunks of four
// folded texels and two of weights feed 64 FMAs.  The chunks of a row are
// stored even ones first, so that the threads of a row, two chunks apart,
// read neighbouring ones (no bank conflict).  A group's sum of a row is FP32
// and is added to an FP32 pair (two-sum: some 48 bits, FP32 rate).
// 1024^2 texels, R = 77: 1.09 -> 0.745 ms.
constexpr int kFoldTX = 64, kFoldTY = 16, kFoldOut = 8;
constexpr int kFoldGroup = (kFoldTX / kFoldOut) * kFoldTY;
constexpr int kFoldSlots = kFoldTY + 1;
constexpr int kFoldMin = 64;  // smallest R folded

// chunks of either parity in a row (two beyond the last tap's), floats of a
// row of weights
__host__ __device__ __forceinline__ int fold_half(int R) {
  return (kFoldTX + 2 * fs_ra(R) + 16) / 8 + 1;
}
__host__ __device__ __forceinline__ int fold_wn(int R) {
  return 2 * fs_ra(R) + 16;
}

// (hi, lo) += v
__device__ __forceinline__ void two_add(float &hi, float &lo, float v) {
  const float t = __fadd_rn(hi, v);
  const float z = __fsub_rn(t, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)),
                               __fsub_rn(v, z)));
  hi = t;
}

// (NL: values a thread stages per dy, at most)
template <int G, int NL>
__global__ void __launch_bounds__(kFoldGroup *G, G == 2 ? 3 : 1)
    k_fs_fold(const float *__restrict__ A, int npix, double L, int R,
              const float *__restrict__ W, const int *__restrict__ rowhw,
              float *__restrict__ out) {
  extern __shared__ __align__(16) float fs_smem[];
  const int Ra = fs_ra(R), half = fold_half(R), wn = fold_wn(R);
  const int pitch = 8 * half, width = kFoldTX + 2 * Ra + 16;
  float *s_up = fs_smem;                        // [17][pitch]
  float *s_dn = s_up + kFoldSlots * pitch;      // [17][pitch]
  float *s_w = s_dn + kFoldSlots * pitch;       // [2][wn]
  const int grp = threadIdx.x / kFoldGroup;
  const int tx = threadIdx.x % (kFoldTX / kFoldOut);
  const int ty = threadIdx.x % kFoldGroup / (kFoldTX / kFoldOut);
  const int x0 = blockIdx.x * kFoldTX, y0 = blockIdx.y * kFoldTY;
  const float Lf = (float)L, dltf = (float)((2.0 * L) / (double)npix);
  auto texel = [&](int c, int y) {
    const int x = x0 - Ra + c;
    return (x >= 0 && x < npix && y >= 0 && y < npix)
               ? __ldg(&A[(size_t)y * npix + x])
               : pspl_at(x, y, Lf, dltf);
  };
  auto place = [&](int c) {  // column c of a row: even chunks first
    return (((c >> 2) & 1) * half + (c >> 3)) * 4 + (c & 3);
  };
  auto weight = [&](int t, int dy) {
    const int dx = t - Ra;
    return (dx >= -R && dx <= R && dy <= R)
               ? __ldg(&W[(size_t)(dy + R) * (2 * R + 1) + (dx + R)])
               : 0.f;
  };
  for (int r = 0; r < kFoldTY; ++r)
    for (int c = threadIdx.x; c < width; c += (kFoldGroup * G)) {
      const float v = 0.5f * texel(c, y0 + r);
      s_up[r * pitch + place(c)] = v;
      s_dn[r * pitch + place(c)] = v;
    }
  for (int t = threadIdx.x; t < wn; t += (kFoldGroup * G)) s_w[t] = 2.f * weight(t, 0);
  float hi[kFoldOut], lo[kFoldOut];
#pragma unroll
  for (int k = 0; k < kFoldOut; ++k) hi[k] = lo[k] = 0.f;
  // slots of output row ty's rows y + dy and y - dy, and of the new rows
  int up = ty, dn = ty, new_up = kFoldTY, new_dn = kFoldSlots - 1;
  int hw = rowhw[R];
  __syncthreads();
  for (int dy = 0; dy <= R && hw >= 0; ++dy) {
    const int hw_next = dy < R ? __ldg(&rowhw[dy + 1 + R]) : -1;
    float next[NL];
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int e = threadIdx.x + i * (kFoldGroup * G);
      if (e < width)
        next[i] = texel(e, y0 + kFoldTY + dy);
      else if (e < 2 * width)
        next[i] = texel(e - width, y0 - dy - 1);
      else if (e < 2 * width + wn)
        next[i] = weight(e - 2 * width, dy + 1);
    }
    // taps dx = t - Ra for t in [Ra - hw, Ra + hw], in pairs p of chunks
    // (eight taps, zero weights beyond the row); output k of tap t is the
    // folded texel 8 tx + t + k
    const int p0 = (Ra - hw) >> 3, np = ((Ra + hw) >> 3) + 1 - p0;
    const int pa = p0 + np * grp / G, pb = p0 + np * (grp + 1) / G;
    if (pa < pb) {
      const float4 *u =
          reinterpret_cast<const float4 *>(s_up + up * pitch) + tx + pa;
      const float4 *d =
          reinterpret_cast<const float4 *>(s_dn + dn * pitch) + tx + pa;
      const float4 *w4 =
          reinterpret_cast<const float4 *>(s_w + (dy & 1) * wn) + 2 * pa;
      const float both = dy > 0 ? 1.f : 0.f;  // dy = 0: the row once
      auto fold = [&](int o) {
        const float4 a = u[o], b = d[o];
        return make_float4(__fmaf_rn(both, b.x, a.x),
                           __fmaf_rn(both, b.y, a.y),
                           __fmaf_rn(both, b.z, a.z),
                           __fmaf_rn(both, b.w, a.w));
      };
      float rs[kFoldOut];
#pragma unroll
      for (int k = 0; k < kFoldOut; ++k) rs[k] = 0.f;
      float4 c0 = fold(0), c1 = fold(half);
#pragma unroll 2
      for (int p = pa; p < pb; ++p, w4 += 2) {
        ++u;
        ++d;
        const float4 c2 = fold(0), c3 = fold(half);
        const float4 wa = w4[0], wb = w4[1];
        const float v[16] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w,
                             c2.x, c2.y, c2.z, c2.w, c3.x, c3.y, c3.z, c3.w};
        const float ww[8] = {wa.x, wa.y, wa.z, wa.w,
                             wb.x, wb.y, wb.z, wb.w};
#pragma unroll
        for (int o = 0; o < 8; ++o)
#pragma unroll
          for (int k = 0; k < kFoldOut; ++k)
            rs[k] = __fmaf_rn(ww[o], v[o + k], rs[k]);
        c0 = c2;
        c1 = c3;
      }
#pragma unroll
      for (int k = 0; k < kFoldOut; ++k) two_add(hi[k], lo[k], rs[k]);
    }
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int e = threadIdx.x + i * (kFoldGroup * G);
      if (e < width)
        s_up[new_up * pitch + place(e)] = 0.5f * next[i];
      else if (e < 2 * width)
        s_dn[new_dn * pitch + place(e - width)] = 0.5f * next[i];
      else if (e < 2 * width + wn)
        s_w[((dy + 1) & 1) * wn + e - 2 * width] = 2.f * next[i];
    }
    hw = hw_next;
    up = up + 1 == kFoldSlots ? 0 : up + 1;
    new_up = new_up + 1 == kFoldSlots ? 0 : new_up + 1;
    dn = dn == 0 ? kFoldSlots - 1 : dn - 1;
    new_dn = new_dn == 0 ? kFoldSlots - 1 : new_dn - 1;
    __syncthreads();
  }
  // the other groups' sums
  float *s_sum = fs_smem;
  if (grp > 0)
#pragma unroll
    for (int k = 0; k < kFoldOut; ++k) {
      float *q = s_sum + 2 * ((grp - 1) * kFoldOut + k) * kFoldGroup +
                 threadIdx.x % kFoldGroup;
      q[0] = hi[k];
      q[kFoldGroup] = lo[k];
    }
  __syncthreads();
  if (grp > 0) return;
  const int y = y0 + ty;
#pragma unroll
  for (int k = 0; k < kFoldOut; ++k) {
    for (int g = 0; g < G - 1; ++g) {
      const float *q = s_sum + 2 * (g * kFoldOut + k) * kFoldGroup +
                       threadIdx.x;
      two_add(hi[k], lo[k], q[0]);
      lo[k] = __fadd_rn(lo[k], q[kFoldGroup]);
    }
    const int x = x0 + kFoldOut * tx + k;
    if (x < npix && y < npix)  // (lo of an infinite sum: NaN)
      out[(size_t)y * npix + x] =
          isfinite(hi[k]) ? __fadd_rn(hi[k], lo[k]) : hi[k];
  }
}

// Source profile integrated over texel (dx, dy), |dx|, |dy| <= R, on
// kSub x kSub midpoint points (unnormalised): the octant 0 <= dy <= dx, one
// thread per row of points (eight to a texel), written to its eight images.
constexpr int kFsSub = 8;
__global__ void k_fs_weights(double rho, double gamma, int R,
                             double *__restrict__ w) {
  const int side = 2 * R + 1;
  const int n = (R + 1) * (R + 1) * kFsSub;
  const double ir2 = 1.0 / (rho * rho);
  for (int k0 = blockIdx.x * blockDim.x; k0 < n; k0 += gridDim.x * blockDim.x) {
    const int k = k0 + threadIdx.x;  // (n is a multiple of 8)
    const int b = k % kFsSub, dy = k / kFsSub / (R + 1),
              dx = k / kFsSub % (R + 1);
    double acc = 0.0;
    if (k < n && dy <= dx) {
      const double y = dy - 0.5 + (b + 0.5) / kFsSub;
      for (int a = 0; a < kFsSub; ++a) {
        const double x = dx - 0.5 + (a + 0.5) / kFsSub;
        const double u2 = (x * x + y * y) * ir2;
        if (u2 < 1.0) acc += 1.0 - gamma * (1.0 - 1.5 * sqrt(1.0 - u2));
      }
    }
    for (int o = 1; o < kFsSub; o <<= 1)
      acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (k < n && dy <= dx) {  // lane b writes image b
      const int u = b & 4 ? dy : dx, v = b & 4 ? dx : dy;
      const int x = R + (b & 1 ? -u : u), y = R + (b & 2 ? -v : v);
      w[(size_t)y * side + x] = acc;
    }
  }
}

// Sums of the rows of w, then the weights as the convolution reads them:
// normalised, rounded to FP32, and the half-width of every row (-1: empty).
// A source that reaches no sample point is its centre texel alone.
__device__ __forceinline__ double fs_block_sum(double v, double *s_red) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += s_red[k];
  __syncthreads();
  return t;
}
__global__ void __launch_bounds__(128)
    k_fs_rows(const double *__restrict__ w, int side,
              double *__restrict__ rows) {
  __shared__ double s_red[4];
  double v = 0.0;
  for (int k = threadIdx.x; k < side; k += blockDim.x)
    v += w[(size_t)blockIdx.x * side + k];
  v = fs_block_sum(v, s_red);
  if (threadIdx.x == 0) rows[blockIdx.x] = v;
}
__global__ void __launch_bounds__(128)
    k_fs_norm(const double *__restrict__ w, const double *__restrict__ rows,
              int side, float *__restrict__ wf, int *__restrict__ hw) {
  __shared__ double s_red[4];
  __shared__ int s_hw;
  if (threadIdx.x == 0) s_hw = -1;
  double v = 0.0;
  for (int k = threadIdx.x; k < side; k += blockDim.x) v += rows[k];
  const double tot = fs_block_sum(v, s_red);
  const int R = side / 2, y = blockIdx.x;
  int m = -1;
  for (int k = threadIdx.x; k < side; k += blockDim.x) {
    const double u = tot > 0.0 ? w[(size_t)y * side + k] / tot
                               : (k == R && y == R ? 1.0 : 0.0);
    wf[(size_t)y * side + k] = (float)u;
    if (u != 0.0) m = max(m, abs(k - R));
  }
  if (m >= 0) atomicMax(&s_hw, m);
  __syncthreads();
  if (threadIdx.x == 0) hw[y] = s_hw;
}

}  // namespace

cudaError_t launch_fs_weights(double rho_px, double gamma, int R, double *w,
                              double *rows, float *wf, int *hw,
                              cudaStream_t st) {
  const long long n = (long long)(R + 1) * (R + 1) * kFsSub;
  long long blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  const int side = 2 * R + 1;
  k_fs_weights<<<(unsigned)blocks, 256, 0, st>>>(rho_px, gamma, R, w);
  k_fs_rows<<<side, 128, 0, st>>>(w, side, rows);
  k_fs_norm<<<side, 128, 0, st>>>(w, rows, side, wf, hw);
  return cudaGetLastError();
}

size_t fs_smem_bytes(int R) {
  return sizeof(float) *
         ((size_t)kFsTY * fs_width(R) + 2 * (size_t)fs_ra(R) + 4);
}

static size_t fold_smem_bytes(int R) {
  return sizeof(float) * ((size_t)2 * kFoldSlots * 8 * fold_half(R) +
                          2 * (size_t)fold_wn(R));
}

template <int G, int NL>
static cudaError_t launch_fold(const float *A, int npix, double L, int R,
                               const float *W, const int *rowhw, float *out,
                               cudaStream_t st) {
  const size_t smem = fold_smem_bytes(R);
  const cudaError_t e = raise_smem(k_fs_fold<G, NL>);
  if (e != cudaSuccess) return e;
  const dim3 grid((npix + kFoldTX - 1) / kFoldTX,
                  (npix + kFoldTY - 1) / kFoldTY);
  k_fs_fold<G, NL><<<grid, kFoldGroup * G, smem, st>>>(A, npix, L, R, W,
                                                       rowhw, out);
  return cudaGetLastError();
}

cudaError_t launch_fs_conv(const float *A, int npix, double L, int R,
                           const float *W, const int *rowhw, float *out,
                           cudaStream_t st) {
  // folded from kFoldMin on (small sources: the unfolded kernel is bound by
  // its tiles' halo, and its one-row sums are the more exact) while the rows
  // fit shared memory and a thread's loads its registers
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int loads = 2 * (kFoldTX + 2 * fs_ra(R) + 16) + fold_wn(R);
  if (R >= kFoldMin && fold_smem_bytes(R) <= (size_t)optin) {
    if (loads <= 2 * 4 * kFoldGroup)
      return launch_fold<2, 4>(A, npix, L, R, W, rowhw, out, st);
    if (loads <= 4 * 4 * kFoldGroup)
      return launch_fold<4, 4>(A, npix, L, R, W, rowhw, out, st);
    if (loads <= 4 * 8 * kFoldGroup)
      return launch_fold<4, 8>(A, npix, L, R, W, rowhw, out, st);
  }
  const size_t smem = fs_smem_bytes(R);
  const cudaError_t e = raise_smem(k_fs_conv);
  if (e != cudaSuccess) return e;
  dim3 grid((npix + kFsTX - 1) / kFsTX, (npix + kFsTY - 1) / kFsTY);
  k_fs_conv<<<grid, kFsThreads, smem, st>>>(A, npix, L, R, W, rowhw, out);
  return cudaGetLastError();
}

}  // namespace morse
