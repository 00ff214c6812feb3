// rm_normals.cu -- rm_depth_normals: surface normals of depth images (Eq. 2, Sec. V).
//
// Gaussian smoothing as a normalised convolution (weighted sums of the valid depths and of their
// weights, along the rows, then down the columns) and the normals N = a x b with a = (0, s_y, dz/dy),
// b = (s_x, 0, dz/dx) by central differences of the smoothed depth S, fused. Each depth and class byte
// is read about once from HBM and each normal written once (17 bytes per pixel). One instantiation per
// radius, so the taps unroll with their weights in registers. Two kernels that add and divide in the
// same order and agree bit for bit:
//   k_depth_normals       many pixels: one warp per (62-column strip, chunk of rows, image) walks down
//                         its strip without block barriers
//   k_depth_normals_tile  few pixels: one CTA per (64x16 output tile, image)
#include <cfloat>
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <string>
#include <type_traits>

#include "rendermap.h"
#include "rm_kernels.cuh"

namespace {

constexpr int kMaxR = 16;              // Gaussian radius ceil(3 sigma) for sigma <= 5
constexpr int kCols = 64;              // smoothed columns of a strip, two per lane
constexpr int kOut = kCols - 2;        // its output columns
constexpr int kRows = 4;               // rows per step
constexpr int kWarpsN = 4;             // warps (strips) per CTA
constexpr long long kNormalWarps = 3040;  // 152 SMs x 20 resident

struct NormalArgs {
  const float *depth;
  const uint8_t *cls;
  float *normals;
  float *smoothed;   // optional
  float *blur;       // optional: S where valid, else the input depth
  int W, H, r, metric;
  int strips, chunks, rows;  // strips across, chunks down an image, output rows of a chunk
  long long n_warps;         // strips * chunks * images
  float ifx, ify;    // 1 / fx, 1 / fy
  float den_all;     // the weight sum where every pixel of the window is valid, summed as the kernels do
  float g[kMaxR + 1];
};

// A staged pixel as (depth, weight), zero where invalid.
__device__ __forceinline__ float2 depth_pair(float d, int c) {
  const bool ok = c == 0 && fabsf(d) <= FLT_MAX;
  return make_float2(ok ? d : 0.0f, ok ? 1.0f : 0.0f);
}

// The normal at smoothed depth s between its neighbours left, right, up and down. S is NaN at invalid
// pixels and outside the image, so an undefined difference makes the normal NaN by itself; only an
// invalid centre needs asking for.
__device__ __forceinline__ float3 eq2_normal(const NormalArgs &a, float s, float sl, float sr, float su, float sd) {
  const float zx = 0.5f * (sr - sl), zy = 0.5f * (sd - su);
  const float sx = a.metric ? s * a.ifx : 1.0f, sy = a.metric ? s * a.ify : 1.0f;
  // a = (0, sy, zy), b = (sx, 0, zx), N = a x b
  const float q0 = sy * zx, q1 = zy * sx, q2 = -sy * sx;
  float inv = rsqrtf(q0 * q0 + q1 * q1 + q2 * q2);
  if (isnan(s)) inv = __builtin_nanf("");
  return make_float3(q0 * inv, q1 * inv, q2 * inv);
}

// ------------------------------------------------------------------ strips (many pixels)
//
// A warp walks down its strip four rows at a time. Each row's depths are staged in shared memory as
// (depth, weight) pairs with a halo of the Gaussian's radius; a lane smooths two adjacent columns
// along the row, sums and weight sums together in packed FP32 pairs, and keeps the result in its own
// ring of the last rows; four smoothed rows then come from one pass down the ring, and the normals
// from the smoothed rows in registers, the columns beside a lane's own by shuffle. Rows are not
// convolved twice and only 12 of 74 columns (radius 5) and the chunk's first and last rows are halo.
// Bound by the shared-memory pipe (0.76 of its peak: about 60 wavefronts a row of 64 columns, two
// fifths of them the row windows) beside instruction issue (0.66). 64 images of 640x480 at radius 5:
// 146 us, where the tiles below take 229 and 1.9 times the instructions.

// a * b + c on both halves, each rounded as one fused multiply-add.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// One warp's shared memory: the step's staged rows, the ring of horizontal sums (a lane's two
// columns side by side, private to it) and one row of normals on its way out.
template <int R>
struct StripSmem {
  static constexpr int kRing = (2 * R + kRows + kRows - 1) / kRows * kRows;  // whole steps
  float4 ring[kRing][32];
  alignas(16) float2 z[kRows][kCols + 2 * R];
  alignas(8) float out[3 * kCols];
};

template <int R>
__global__ void __launch_bounds__(32 * kWarpsN) k_depth_normals(NormalArgs a) {
  extern __shared__ float4 smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  StripSmem<R> &sm = reinterpret_cast<StripSmem<R> *>(smem_raw)[warp];
  const long long job = (long long)blockIdx.x * kWarpsN + warp;
  if (job >= a.n_warps) return;
  const int strip = (int)(job % a.strips), chunk = (int)(job / a.strips % a.chunks);
  const long long img = job / ((long long)a.strips * a.chunks), P = (long long)a.W * a.H;
  const float *dimg = a.depth + img * P;
  const uint8_t *cimg = a.cls + img * P;
  const int xs = strip * kOut - 1;                 // image column of smoothed column 0
  const int y_out = chunk * a.rows, y_end = min(y_out + a.rows, a.H);
  float2 g[R + 1];
#pragma unroll
  for (int k = 0; k <= R; ++k) g[k] = make_float2(a.g[k], a.g[k]);
  constexpr float kNan = __builtin_nanf("");
  // this lane's columns: two of its own and one of the halo
  const int x0 = xs + 2 * lane, hc = lane < R ? lane : kCols + lane, xh = xs - R + hc;
  const bool in0 = x0 >= 0 && x0 < a.W, in1 = x0 + 1 >= 0 && x0 + 1 < a.W;
  const bool inh = lane < 2 * R && xh >= 0 && xh < a.W;
  float zd[kRows][3];
  int zc[kRows][3];
  const int y_first = y_out - 1 - R;
  const float *dp = dimg + (long long)y_first * a.W;  // the next step's first row
  const uint8_t *cp = cimg + (long long)y_first * a.W;
  auto load = [&](int y0) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const bool iy = y0 + r >= 0 && y0 + r < a.H;
      zd[r][0] = zd[r][1] = zd[r][2] = 0.0f;
      zc[r][0] = zc[r][1] = zc[r][2] = 1;
      if (iy) {
        if (in0) zd[r][0] = __ldg(dp + x0), zc[r][0] = __ldg(cp + x0);
        if (in1) zd[r][1] = __ldg(dp + x0 + 1), zc[r][1] = __ldg(cp + x0 + 1);
        if (inh) zd[r][2] = __ldg(dp + xh), zc[r][2] = __ldg(cp + xh);
      }
      dp += a.W;
      cp += a.W;
    }
  };
  const int n_out = 3 * min(kOut, a.W - (xs + 1));
  long long at_out = img * P + (long long)y_out * a.W;  // the next output row
  unsigned long long v0 = 0, v1 = 0;               // validity of the own columns, last row in bit 0
  float s0a = kNan, s1a = kNan, s0b = kNan, s1b = kNan;  // smoothed rows before the step's (a: two before)
  int slot = 0;                                    // ring slot of the step's first row
  load(y_first);
  for (int y0 = y_first; y0 <= y_end + R; y0 += kRows) {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const float2 p0 = depth_pair(zd[r][0], zc[r][0]), p1 = depth_pair(zd[r][1], zc[r][1]),
                   ph = depth_pair(zd[r][2], zc[r][2]);
      sm.z[r][R + 2 * lane] = p0;
      sm.z[r][R + 2 * lane + 1] = p1;
      if (lane < 2 * R) sm.z[r][hc] = ph;
      v0 = v0 << 1 | (p0.y != 0.0f);
      v1 = v1 << 1 | (p1.y != 0.0f);
    }
    __syncwarp();
    if (y0 + kRows <= y_end + R) load(y0 + kRows);
    // along the rows: staged columns 2 lane .. 2 lane + 2R + 1 hold both columns' windows
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const float4 *w = reinterpret_cast<const float4 *>(&sm.z[r][2 * lane]);
      float2 n0 = make_float2(0.0f, 0.0f), n1 = n0;
#pragma unroll
      for (int t = 0; t <= R; ++t) {
        const float4 q = w[t];
        const float2 lo = make_float2(q.x, q.y), hi = make_float2(q.z, q.w);
        const int k = 2 * t;                       // lo is tap k of column 0, hi tap k of column 1
        n0 = fma2(g[k < R ? R - k : k - R], lo, n0);
        if (k + 1 <= 2 * R) n0 = fma2(g[k + 1 < R ? R - k - 1 : k + 1 - R], hi, n0);
        if (k >= 1) n1 = fma2(g[k - 1 < R ? R - k + 1 : k - 1 - R], lo, n1);
        n1 = fma2(g[k < R ? R - k : k - R], hi, n1);
      }
      sm.ring[slot + r][lane] = make_float4(n0.x, n0.y, n1.x, n1.y);
    }
    // down the ring: smoothed rows y0 - R .. y0 - R + 3 from rows y0 - 2R .. y0 + 3
    float2 m0[kRows], m1[kRows];
#pragma unroll
    for (int j = 0; j < kRows; ++j) m0[j] = m1[j] = make_float2(0.0f, 0.0f);
    int at = slot - 2 * R;
    if (at < 0) at += StripSmem<R>::kRing;
#pragma unroll
    for (int t = 0; t < 2 * R + kRows; ++t) {
      const float4 q = sm.ring[at][lane];
      if (++at == StripSmem<R>::kRing) at = 0;
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        const int d = t - j;
        if (d >= 0 && d <= 2 * R) {
          const float2 w = g[d < R ? R - d : d - R];
          m0[j] = fma2(w, make_float2(q.x, q.y), m0[j]);
          m1[j] = fma2(w, make_float2(q.z, q.w), m1[j]);
        }
      }
    }
    slot += kRows;
    if (slot == StripSmem<R>::kRing) slot = 0;
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      // the smoothed row ys (centres valid), then the normals of the row above it
      const int ys = y0 - R + j, y = ys - 1;
      const bool c0 = v0 >> (R + kRows - 1 - j) & 1, c1 = v1 >> (R + kRows - 1 - j) & 1;
      const float s0 = c0 ? m0[j].x / m0[j].y : kNan, s1 = c1 ? m1[j].x / m1[j].y : kNan;
      const float left = __shfl_up_sync(0xffffffffu, s1b, 1), right = __shfl_down_sync(0xffffffffu, s0b, 1);
      if (y >= y_out && y < y_end) {
        if (a.smoothed || a.blur) {
          const bool w0 = lane > 0 && x0 < a.W, w1 = lane < 31 && x0 + 1 < a.W;
          if (a.smoothed) {
            if (w0) a.smoothed[at_out + x0] = s0b;
            if (w1) a.smoothed[at_out + x0 + 1] = s1b;
          }
          if (a.blur) {
            if (w0) a.blur[at_out + x0] = isnan(s0b) ? a.depth[at_out + x0] : s0b;
            if (w1) a.blur[at_out + x0 + 1] = isnan(s1b) ? a.depth[at_out + x0 + 1] : s1b;
          }
        }
        if (a.normals) {
          float2 *o = reinterpret_cast<float2 *>(sm.out) + 3 * lane;
          const float3 p = eq2_normal(a, s0b, left, s1b, s0a, s0), q = eq2_normal(a, s1b, s0b, right, s1a, s1);
          o[0] = make_float2(p.x, p.y);
          o[1] = make_float2(p.z, q.x);
          o[2] = make_float2(q.y, q.z);
          __syncwarp();
          float *dst = a.normals + 3 * (at_out + xs + 1) + lane;
#pragma unroll
          for (int k = 0; k < 6; ++k)
            if (lane + 32 * k < n_out) dst[32 * k] = sm.out[3 + lane + 32 * k];
          __syncwarp();
        }
        at_out += a.W;
      }
      s0a = s0b;
      s1a = s1b;
      s0b = s0;
      s1b = s1;
    }
  }
}

// ------------------------------------------------------------------ tiles (few pixels)
//
// A strip's warp is a long chain: its chunk is no shorter than the halo that it reads besides, and
// with few pixels there are too few warps to hide it. Here one CTA stages a tile's depths and weights
// with a halo of radius + 1, smooths along the rows (four outputs a thread) and down the columns
// (six), and takes the differences of the smoothed tile. Bound by latency: a load, two passes and two
// barriers. One image of 640x480 with strips and with tiles: radius 2 8.4 and 4.6 us, 5 14.1 and 5.7,
// 8 21.6 and 7.3, 15 43.2 and 10.5.

constexpr int kTW = 64, kTH = 16;      // output tile
constexpr int kSW = kTW + 2;           // smoothed region (tile plus a one-pixel ring)
constexpr int kSH = kTH + 2;
constexpr int kTileThreads = 256;
constexpr int kHG = 4;                 // along the rows: outputs per thread
constexpr int kVG = 6;                 // down the columns: outputs per thread
// Below this many pixels in all the tiles are faster, at any radius but 0: at 1.2 M pixels strips take
// 1.25 to 1.6 times as long (4 images of 640x480; 64 of 160x120, 0.95 to 1.2), at 2.1 M to 2.5 M 0.7 to
// 1.3 (widths and radii either way), at 4.9 M 0.7 to 1.1. At radius 0 strips take 0.75 to 1.15 times
// as long from one small image on.
constexpr long long kTilePixels = 1ll << 21;

// The tables' row strides are odd: the pass along the rows goes down their columns with consecutive
// threads on consecutive rows, and 32 consecutive rows then fall in 32 distinct banks.
__host__ __device__ constexpr int odd_stride(int n) { return n | 1; }
template <int R>
struct TileShape {
  static constexpr int kW = kSW + 2 * R, kH = kSH + 2 * R, kStride = odd_stride(kW);  // staged pixels
  static constexpr int kSumStride = odd_stride(kSW);
  static constexpr size_t kBytes = sizeof(float) * (2 * kH * kStride + 2 * kH * kSumStride + kSH * kSW);
};

template <int R>
__global__ void __launch_bounds__(kTileThreads) k_depth_normals_tile(NormalArgs a) {
  extern __shared__ float4 smem_raw[];
  using Shape = TileShape<R>;
  constexpr int dw = Shape::kW, dh = Shape::kH, dws = Shape::kStride, hs = Shape::kSumStride;
  float *zv = reinterpret_cast<float *>(smem_raw);  // [dh][dws]: valid ? z : 0
  float *zw = zv + dh * dws;                        // [dh][dws]: valid ? 1 : 0
  float *hn = zw + dh * dws;                        // [dh][hs]: sums of zv along the rows
  float *hd = hn + dh * hs;                         // [dh][hs]: sums of zw
  float *sS = hd + dh * hs;                         // [kSH][kSW]: smoothed depth
  const int tid = threadIdx.x;
  float g[R + 1];
#pragma unroll
  for (int k = 0; k <= R; ++k) g[k] = a.g[k];
  const int ntx = (a.W + kTW - 1) / kTW;
  const int ox = (blockIdx.x % ntx) * kTW, oy = (blockIdx.x / ntx) * kTH;
  const int x0 = ox - 1 - R, y0 = oy - 1 - R;  // image coordinates of zv[0]
  const long long P = (long long)a.W * a.H, img = blockIdx.y;
  const float *dimg = a.depth + img * P;
  const uint8_t *cimg = a.cls + img * P;
  // stage, four loads in flight a thread; whether every staged pixel is valid is the common case away
  // from holes and the image border
  constexpr int n_st = dw * dh;
  bool mine_valid = true;
  for (int k0 = tid; k0 < n_st; k0 += 4 * kTileThreads) {
    float dv[4];
    int cv[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int k = k0 + m * kTileThreads, x = x0 + k % dw, y = y0 + k / dw;
      dv[m] = 0.0f;
      cv[m] = 1;
      if (k < n_st && x >= 0 && x < a.W && y >= 0 && y < a.H) {
        const long long p = (long long)y * a.W + x;
        dv[m] = __ldg(dimg + p);
        cv[m] = __ldg(cimg + p);
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int k = k0 + m * kTileThreads;
      if (k < n_st) {
        const float2 z = depth_pair(dv[m], cv[m]);
        const int at = (k / dw) * dws + k % dw;
        mine_valid = mine_valid && z.y != 0.0f;
        zv[at] = z.x;
        zw[at] = z.y;
      }
    }
  }
  const bool all_valid = __syncthreads_and(mine_valid);
  // along the rows, then down the columns: a value is loaded once and added to every output whose
  // window holds it; the weight sums only where a staged pixel is invalid
  auto smooth = [&](auto all) {
    constexpr bool kAll = decltype(all)::value;
    constexpr int h_groups = (kSW + kHG - 1) / kHG, v_groups = (kSH + kVG - 1) / kVG;
    for (int it = tid; it < dh * h_groups; it += kTileThreads) {
      const int v = it % dh, u0 = (it / dh) * kHG;
      float num[kHG], den[kHG];
#pragma unroll
      for (int j = 0; j < kHG; ++j) num[j] = den[j] = 0.0f;
      const float *row = zv + v * dws + u0, *roww = zw + v * dws + u0;
#pragma unroll
      for (int t = 0; t < 2 * R + kHG; ++t) {
        const bool in = u0 + t < dw;
        const float z = in ? row[t] : 0.0f, zok = !kAll && in ? roww[t] : 0.0f;
#pragma unroll
        for (int j = 0; j < kHG; ++j) {
          const int d = t - j;
          if (d >= 0 && d <= 2 * R) {
            const float w = g[d < R ? R - d : d - R];
            num[j] = fmaf(w, z, num[j]);
            if (!kAll) den[j] = fmaf(w, zok, den[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kHG; ++j)
        if (u0 + j < kSW) {
          hn[v * hs + u0 + j] = num[j];
          if (!kAll) hd[v * hs + u0 + j] = den[j];
        }
    }
    __syncthreads();
    for (int it = tid; it < kSW * v_groups; it += kTileThreads) {
      const int u = it % kSW, v0 = (it / kSW) * kVG;
      float num[kVG], den[kVG];
#pragma unroll
      for (int j = 0; j < kVG; ++j) num[j] = den[j] = 0.0f;
#pragma unroll
      for (int t = 0; t < 2 * R + kVG; ++t) {
        const bool in = v0 + t < dh;
        const float hz = in ? hn[(v0 + t) * hs + u] : 0.0f, hw = !kAll && in ? hd[(v0 + t) * hs + u] : 0.0f;
#pragma unroll
        for (int j = 0; j < kVG; ++j) {
          const int d = t - j;
          if (d >= 0 && d <= 2 * R) {
            const float w = g[d < R ? R - d : d - R];
            num[j] = fmaf(w, hz, num[j]);
            if (!kAll) den[j] = fmaf(w, hw, den[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kVG; ++j) {
        const int v = v0 + j;
        if (v < kSH) {
          const bool centre = kAll || zw[(v + R) * dws + (u + R)] != 0.0f;
          sS[v * kSW + u] = centre ? num[j] / (kAll ? a.den_all : den[j]) : __builtin_nanf("");
        }
      }
    }
  };
  if (all_valid) smooth(std::true_type{});
  else smooth(std::false_type{});
  __syncthreads();
  for (int k = tid; k < kTW * kTH; k += kTileThreads) {
    const int u = k % kTW + 1, v = k / kTW + 1, x = ox + u - 1, y = oy + v - 1;
    if (x >= a.W || y >= a.H) continue;
    const long long p = img * P + (long long)y * a.W + x;
    const float *c = sS + v * kSW + u;
    if (a.smoothed) a.smoothed[p] = *c;
    if (a.blur) a.blur[p] = isnan(*c) ? a.depth[p] : *c;
    if (!a.normals) continue;
    const float3 n = eq2_normal(a, c[0], c[-1], c[1], c[-kSW], c[kSW]);
    a.normals[3 * p] = n.x;
    a.normals[3 * p + 1] = n.y;
    a.normals[3 * p + 2] = n.z;
  }
}

template <int R>
cudaError_t launch_normals_r(const NormalArgs &a, int n, cudaStream_t s) {
  // the larger radii need more than the default 48 KB (set on the current device)
  if constexpr (R > 0) {
    if ((long long)a.W * a.H * n < kTilePixels) {
      const size_t sm = TileShape<R>::kBytes;
      cudaError_t e = cudaFuncSetAttribute(k_depth_normals_tile<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
      const int tiles = ((a.W + kTW - 1) / kTW) * ((a.H + kTH - 1) / kTH);
      k_depth_normals_tile<R><<<dim3(tiles, n), kTileThreads, sm, s>>>(a);
      return cudaGetLastError();
    }
  }
  const size_t sm = sizeof(StripSmem<R>) * kWarpsN;
  cudaError_t e = cudaFuncSetAttribute(k_depth_normals<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_depth_normals<R><<<(unsigned)((a.n_warps + kWarpsN - 1) / kWarpsN), 32 * kWarpsN, sm, s>>>(a);
  return cudaGetLastError();
}

template <int R>
cudaError_t launch_normals(const NormalArgs &a, int n, cudaStream_t s) {
  if (a.r == R) return launch_normals_r<R>(a, n, s);
  if constexpr (R < kMaxR) return launch_normals<R + 1>(a, n, s);
  return cudaErrorInvalidValue;
}

bool dn_on_device(const void *p) {
  if (!p) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

rm_status dn_fail(rm_status s, const std::string &m) {
  rmapi::set_error(m);
  return s;
}

// Shared driver of rm_depth_normals and rm_depth_blur; any of the three outputs may be NULL.
rm_status run_normals(const rm_intrinsics *intr, int32_t n, const float *depth, const uint8_t *cls,
                      float sigma, int32_t metric, float *normals, float *smoothed, float *blur,
                      void *stream) {
  if (!intr) return dn_fail(RM_EINVAL, "intrinsics are NULL");
  if (n < 0 || intr->width < 0 || intr->height < 0) return dn_fail(RM_EINVAL, "negative size");
  if (n > 65535) return dn_fail(RM_EINVAL, "at most 65535 images per call");
  if (!(sigma >= 0.0f) || sigma > 5.0f) return dn_fail(RM_EINVAL, "sigma must be in [0, 5]");
  if (metric != 0 && metric != 1) return dn_fail(RM_EINVAL, "metric must be 0 or 1");
  if (metric && (intr->model != RM_PINHOLE || !(intr->fx > 0.0f) || !(intr->fy > 0.0f) ||
                 !(intr->fx <= FLT_MAX) || !(intr->fy <= FLT_MAX)))
    return dn_fail(RM_EINVAL, "metric normals need a pinhole camera with finite fx, fy > 0");
  const long long P = (long long)intr->width * intr->height;
  if (n == 0 || P == 0) return RM_OK;
  if (!depth || !cls) return dn_fail(RM_EINVAL, "NULL array");
  if ((long long)n * P > (1LL << 40)) return dn_fail(RM_EINVAL, "too many pixels");
  cudaStream_t s = (cudaStream_t)stream;
  const bool host_d = !dn_on_device(depth), host_c = !dn_on_device(cls);
  const bool host_n = normals && !dn_on_device(normals), host_s = smoothed && !dn_on_device(smoothed);
  const bool host_b = blur && !dn_on_device(blur);
  const size_t np = (size_t)n * P;
  // host arrays are staged through stream-ordered device allocations
  float *d_d = host_d ? nullptr : const_cast<float *>(depth);
  float *d_n = host_n ? nullptr : normals;
  float *d_s = host_s ? nullptr : smoothed;
  float *d_b = host_b ? nullptr : blur;
  uint8_t *d_c = host_c ? nullptr : const_cast<uint8_t *>(cls);
  cudaError_t e = cudaSuccess;
  auto ck = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
  };
  if (host_d) ck(rmapi::scratch_alloc((void **)&d_d, sizeof(float) * np, s));
  if (host_c) ck(rmapi::scratch_alloc((void **)&d_c, np, s));
  if (host_n) ck(rmapi::scratch_alloc((void **)&d_n, sizeof(float) * 3 * np, s));
  if (host_s) ck(rmapi::scratch_alloc((void **)&d_s, sizeof(float) * np, s));
  if (host_b) ck(rmapi::scratch_alloc((void **)&d_b, sizeof(float) * np, s));
  if (e == cudaSuccess && host_d) ck(cudaMemcpyAsync(d_d, depth, sizeof(float) * np, cudaMemcpyHostToDevice, s));
  if (e == cudaSuccess && host_c) ck(cudaMemcpyAsync(d_c, cls, np, cudaMemcpyHostToDevice, s));
  if (e == cudaSuccess) {
    NormalArgs a{};
    a.depth = d_d;
    a.cls = d_c;
    a.normals = d_n;
    a.smoothed = d_s;
    a.blur = d_b;
    a.W = intr->width;
    a.H = intr->height;
    a.r = sigma > 0.0f ? (int)std::ceil(3.0 * (double)sigma) : 0;
    a.metric = metric;
    a.ifx = metric ? 1.0f / intr->fx : 1.0f;
    a.ify = metric ? 1.0f / intr->fy : 1.0f;
    for (int k = 0; k <= kMaxR; ++k)
      a.g[k] = sigma > 0.0f ? (float)std::exp(-(double)(k * k) / (2.0 * (double)sigma * sigma)) : 1.0f;
    float row = 0.0f;
    for (int d = 0; d <= 2 * a.r; ++d) row = std::fmaf(a.g[std::abs(d - a.r)], 1.0f, row);
    for (int d = 0; d <= 2 * a.r; ++d) a.den_all = std::fmaf(a.g[std::abs(d - a.r)], row, a.den_all);
    // chunks of rows: as many warps as are resident at once, but no chunk shorter than the rows that
    // it reads besides its own (64 images of 640x480: 167 us with 2816 warps, 177 with 6336)
    a.strips = (a.W + kOut - 1) / kOut;
    const long long per_row_of_chunks = (long long)a.strips * n;
    const int want = (int)std::max<long long>(1, kNormalWarps / per_row_of_chunks);
    a.rows = std::max((a.H + want - 1) / want, 2 * a.r + 2);
    a.chunks = (a.H + a.rows - 1) / a.rows;
    a.n_warps = per_row_of_chunks * a.chunks;
    ck(launch_normals<0>(a, n, s));
  }
  if (e == cudaSuccess && host_n) ck(cudaMemcpyAsync(normals, d_n, sizeof(float) * 3 * np, cudaMemcpyDeviceToHost, s));
  if (e == cudaSuccess && host_s) ck(cudaMemcpyAsync(smoothed, d_s, sizeof(float) * np, cudaMemcpyDeviceToHost, s));
  if (e == cudaSuccess && host_b) ck(cudaMemcpyAsync(blur, d_b, sizeof(float) * np, cudaMemcpyDeviceToHost, s));
  if (host_d && d_d) cudaFreeAsync(d_d, s);
  if (host_c && d_c) cudaFreeAsync(d_c, s);
  if (host_n && d_n) cudaFreeAsync(d_n, s);
  if (host_s && d_s) cudaFreeAsync(d_s, s);
  if (host_b && d_b) cudaFreeAsync(d_b, s);
  if (e == cudaSuccess && (host_n || host_s || host_b)) ck(cudaStreamSynchronize(s));
  if (e != cudaSuccess) return dn_fail(RM_ECUDA, std::string("rm_depth_normals: ") + cudaGetErrorString(e));
  return RM_OK;
}

// True when the byte ranges [a, a + na) and [b, b + nb) share a byte (NULL overlaps nothing).
bool overlaps(const void *a, size_t na, const void *b, size_t nb) {
  if (!a || !b) return false;
  const char *a0 = static_cast<const char *>(a), *b0 = static_cast<const char *>(b);
  return a0 < b0 + nb && b0 < a0 + na;
}

}  // namespace

extern "C" rm_status rm_depth_normals(const rm_intrinsics *intr, int32_t n, const float *depth,
                                      const uint8_t *cls, float sigma, int32_t metric,
                                      float *normals, float *smoothed, void *stream) {
  if (!normals && n > 0) return dn_fail(RM_EINVAL, "normals is NULL");
  // neighbouring tiles read the inputs' halos while a tile writes its outputs, so no output
  // may share memory with an input or with the other output
  if (intr && n > 0 && intr->width > 0 && intr->height > 0) {
    const size_t np = (size_t)n * intr->width * intr->height;
    const size_t bd = sizeof(float) * np, bc = np, bn = 3 * sizeof(float) * np, bs = sizeof(float) * np;
    if (overlaps(normals, bn, depth, bd) || overlaps(normals, bn, cls, bc))
      return dn_fail(RM_EINVAL, "normals overlaps an input");
    if (overlaps(smoothed, bs, depth, bd) || overlaps(smoothed, bs, cls, bc))
      return dn_fail(RM_EINVAL, "smoothed overlaps an input");
    if (overlaps(normals, bn, smoothed, bs)) return dn_fail(RM_EINVAL, "normals overlaps smoothed");
  }
  return run_normals(intr, n, depth, cls, sigma, metric, normals, smoothed, nullptr, stream);
}

extern "C" rm_status rm_depth_blur(const rm_intrinsics *intr, int32_t n, const float *depth,
                                   const uint8_t *cls, float sigma, float *out, void *stream) {
  if (!out && n > 0) return dn_fail(RM_EINVAL, "out is NULL");
  if (intr && n > 0 && intr->width > 0 && intr->height > 0) {
    const size_t np = (size_t)n * intr->width * intr->height;
    if (overlaps(out, sizeof(float) * np, depth, sizeof(float) * np)) return dn_fail(RM_EINVAL, "out overlaps depth");
    if (overlaps(out, sizeof(float) * np, cls, np)) return dn_fail(RM_EINVAL, "out overlaps cls");
  }
  return run_normals(intr, n, depth, cls, sigma, 0, nullptr, nullptr, out, stream);
}
