// Front end of the tracker: the depth pyramid and the vertex / normal maps the
// coarse-to-fine ICP runs on (the KinectFusion preprocessing the paper builds
// on), and the model-map preparation. One launch covers every pair of a
// batch: blockIdx.z selects the pair.
#include "kf_internal.cuh"

namespace kf {
namespace {

constexpr int kTx = 32, kTy = 8;
// resident front-end blocks per SM the register budget is sized for
#ifndef KF_FE_MINB
#define KF_FE_MINB 6
#endif
// bilateral filter: 1 two vertically adjacent pixels per thread step with
// packed FP32x2 arithmetic; 0 one pixel per step (the same bits either way)
#ifndef KF_FE_PAIRS
#define KF_FE_PAIRS 1
#endif

__device__ __forceinline__ bool valid_depth(float z) { return isfinite(z) && z > 0.f; }

// Model level l = level-0 model maps at pixels (x 2^l, y 2^l), as records; a
// pixel is a hole (NaN vertex and normal) when any component is non-finite or
// the normal is all zero. One launch, each pixel read once and written to every
// level it belongs to; it also brings the pair's descriptor on the device up
// to date (its copy `desc` comes with the launch), which a copy of its own would
// take longer to queue than this kernel runs.
template <class T>
__global__ void __launch_bounds__(kTx* kTy) k_model_prep(const __grid_constant__ PairDesc desc, PairDesc* d_desc,
                                                         const float* Vin, const float* Nin, int w, int h) {
  const int tid = threadIdx.y * kTx + threadIdx.x;
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    constexpr int kWords = sizeof(PairDesc) / sizeof(unsigned long long);
    static_assert(sizeof(PairDesc) % sizeof(unsigned long long) == 0 && kWords <= kTx * kTy, "descriptor size");
    if (tid < kWords)
      reinterpret_cast<unsigned long long*>(d_desc)[tid] = reinterpret_cast<const unsigned long long*>(&desc)[tid];
  }
  const int x = blockIdx.x * kTx + threadIdx.x, y = blockIdx.y * kTy + threadIdx.y;
  if (x >= w || y >= h) return;
  const long src = ((long)y * w + x) * 3;
  const float vx = __ldg(Vin + src), vy = __ldg(Vin + src + 1), vz = __ldg(Vin + src + 2);
  const float nx = __ldg(Nin + src), ny = __ldg(Nin + src + 1), nz = __ldg(Nin + src + 2);
  const bool ok = isfinite(vx) && isfinite(vy) && isfinite(vz) && isfinite(nx) && isfinite(ny) &&
                  isfinite(nz) && (nx != 0.f || ny != 0.f || nz != 0.f);
  const float nan = __int_as_float(0x7fc00000);
  const float4 a = ok ? make_float4(vx, vy, vz, nx) : make_float4(nan, nan, nan, nan);
  const float2 b = ok ? make_float2(ny, nz) : make_float2(nan, nan);
#pragma unroll
  for (int l = 0; l < KF_MAX_LEVELS; ++l) {
    if (l >= desc.levels || ((x | y) & ((1 << l) - 1)) != 0) break;
    const LevelMaps& L = desc.lv[l];
    const int xl = x >> l, yl = y >> l;
    if (xl >= L.mw || yl >= L.mh) break;
    Store<T>::store_a(L.mA, yl * L.mw + xl, a);
    Store<T>::store_b(L.mB, yl * L.mw + xl, b);
  }
}

// ---------------------------------------------------------------------------
// Fused front end: one block owns a 32 x 32 tile of level 0 and the matching
// (32 >> l)^2 tile of every coarser level. It loads the raw depth of its tile
// plus halo into shared memory once, filters a region large enough for every
// level's neighbours, downsamples it level by level in shared memory and
// writes depth, vertex and normal maps:
//  * bilateral (level 0): D'(u) = sum D(u+d) w / sum w over the (2r+1)^2
//    window, w = exp(-|d|^2 / 2 sigma_s^2 - (D(u+d) - D(u))^2 / 2 sigma_r^2),
//    valid neighbours inside the image only, 0 where D(u) is not valid;
//  * level l+1 depth: mean of the valid depths of the 2x2 block within
//    3 sigma_r of the first valid one in scan order (the test in float32:
//    |z - anchor| <= (float)(3 sigma_r)); 0 if the block is empty;
//  * vertex v = z K^-1 (u, v, 1); normal = normalise((v(x+1,y) - v) x
//    (v(x,y+1) - v)) flipped to face the camera; the vertex is stored as NaN
//    where it or its normal is invalid, so the ICP reads one map to decide
//    whether a frame pixel takes part.
// ---------------------------------------------------------------------------
constexpr int kTile = 32;

// side of the level-0 region that is filtered, and of the raw region around it
__host__ __device__ constexpr int region0(int levels) { return ((kTile >> (levels - 1)) + 1) << (levels - 1); }

// Row stride of the raw region's pairs, from its side RR on: half the filtered
// region's side R0 modulo 8, so that a warp whose 32 pixels go on in the
// region's next row of pairs reads the other banks there (without it a third of
// the filter's shared-memory wavefronts were conflicts).
__host__ __device__ constexpr int pair_stride(int R0, int RR) { return RR + (((R0 + 1) / 2 - RR) % 8 + 8) % 8; }

// Calls f(lx, ly) for the cells t = tid, tid + nthr, ... of a w x h region
// in row-major order, stepping the coordinates instead of dividing t.
template <class F>
__device__ __forceinline__ void for_region(int w, int h, int tid, int nthr, F f) {
  const int q = nthr / w, r = nthr - q * w;
  int ly = tid / w, lx = tid - ly * w;
#pragma unroll 1
  while (ly < h) {
    f(lx, ly);
    lx += r;
    ly += q;
    if (lx >= w) {
      lx -= w;
      ++ly;
    }
  }
}

// The vertex of the pixel with (u - c) = (ux, uy) and depth z, and whether it
// has one: x = (u_c z) / f as (u_c z) (1 / f), each product rounded.
__device__ __forceinline__ bool back_project(float ux, float uy, float ifx, float ify, float z, float3& v) {
  v.x = __fmul_rn(__fmul_rn(ux, z), ifx);
  v.y = __fmul_rn(__fmul_rn(uy, z), ify);
  v.z = z;
  return z > 0.f;
}

// Maps of a level's tile x tile pixels from (ox, oy) on. A thread takes kRows
// pixels below one another: the column's coordinates are formed once, and a
// pixel's lower neighbour is the next pixel. The block's threads from kFirst on
// take part. Ds: level depth region of R x R
// whose origin is level pixel (ox, oy).
template <class T, int kTileL, int kRows, int kFirst = 0>
__device__ __forceinline__ void write_maps(const LevelMaps& Lg, const float* Ds, int R, int ox, int oy) {
  // a local copy: the map stores below could alias the descriptor in global
  // memory, which would force its fields to be reloaded for every pixel
  const LevelMaps L = Lg;
  const float nan = __int_as_float(0x7fc00000);
  const float ifx = L.fifx, ify = L.fify;
  const int tid = threadIdx.y * kTx + threadIdx.x - kFirst;
  if (tid < 0 || tid >= kTileL * kTileL / kRows) return;
  const int lx = tid % kTileL, ly0 = tid / kTileL * kRows;
  const int x = ox + lx;
  if (x >= L.fw) return;
  // (float)(x + 1) is (float)x + 1 exactly for image coordinates
  const float fx0 = (float)x, fy0 = (float)(oy + ly0);
  const float ux0 = __fsub_rn(fx0, L.fcx), ux1 = __fsub_rn(fx0 + 1.f, L.fcx);
  const float* D = Ds + ly0 * R + lx;
  const bool right = x + 1 < L.fw;
  float3 v;
  float uy = __fsub_rn(fy0, L.fcy);
  bool ok = back_project(ux0, uy, ifx, ify, D[0], v);
#pragma unroll
  for (int r = 0; r < kRows; ++r, D += R) {
    const int y = oy + ly0 + r;
    if (y >= L.fh) return;
    const float uy1 = __fsub_rn(fy0 + (float)(r + 1), L.fcy);
    float3 v10, v01;
    const bool ok10 = back_project(ux1, uy, ifx, ify, D[1], v10);
    const bool ok01 = back_project(ux0, uy1, ifx, ify, D[R], v01);
    // the decisions (a normal exists; it faces the camera) are float32 with
    // every operation rounded in this order, no contraction: a = v10 - v,
    // b = v01 - v; c = a x b, products rounded, then the difference;
    // l2 = (cx cx + cy cy) + cz cz: a normal iff finite and > 0;
    // s = (cx vx + cy vy) + cz vz > 0 flips it (decided before normalising)
    const float ax = __fsub_rn(v10.x, v.x), ay = __fsub_rn(v10.y, v.y), az = __fsub_rn(v10.z, v.z);
    const float bx = __fsub_rn(v01.x, v.x), by = __fsub_rn(v01.y, v.y), bz = __fsub_rn(v01.z, v.z);
    const float cx = __fsub_rn(__fmul_rn(ay, bz), __fmul_rn(az, by));
    const float cy = __fsub_rn(__fmul_rn(az, bx), __fmul_rn(ax, bz));
    const float cz = __fsub_rn(__fmul_rn(ax, by), __fmul_rn(ay, bx));
    const float len2 = __fadd_rn(__fadd_rn(__fmul_rn(cx, cx), __fmul_rn(cy, cy)), __fmul_rn(cz, cz));
    const float sd = __fadd_rn(__fadd_rn(__fmul_rn(cx, v.x), __fmul_rn(cy, v.y)), __fmul_rn(cz, v.z));
    const bool nok = ok && ok10 && ok01 && right && y + 1 < L.fh && len2 > 0.f && len2 < __int_as_float(0x7f800000);
    const float len = rsqrtf(len2), inv = sd > 0.f ? -len : len;
    const int i = y * L.fw + x;
    L.fdepth[i] = D[0];
    // without a normal (which needs the vertex) both are NaN
    Store<T>::store_a(L.fA, i, nok ? make_float4(v.x, v.y, v.z, cx * inv) : make_float4(nan, nan, nan, nan));
    Store<T>::store_b(L.fB, i, nok ? make_float2(cy * inv, cz * inv) : make_float2(nan, nan));
    v = v01;
    ok = ok01;
    uy = uy1;
  }
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Raw depth that is missing, invalid or outside the image is held as kNoDepth
// in shared memory: its range term (k 1e30 - k z)^2 overflows to +inf, so its
// weight 2^-inf is exactly +0 and it adds nothing (0 * 1e30 = 0), with no
// per-tap test.
constexpr float kNoDepth = 1e30f;

// The filter for two vertically adjacent pixels (cx, cy) and (cx, cy + 1) at
// once: s_pair[y RR + x] holds (D(x, y), D(x, y + 1)), so one 8-byte load
// brings both pixels' neighbour at a tap, and packed FP32x2 fused
// multiply-adds and additions (each lane the scalar operation of
// bilateral_at, in the same order: the same bits) weigh and sum them.
template <int R>
__device__ __forceinline__ float2 bilateral_pair(const float2* s_pair, int RR, int cx, int cy,
                                                 float2 z, const KParams& P) {
  float2 num = make_float2(0.f, 0.f), den = make_float2(0.f, 0.f);
  const float2 k2 = make_float2(P.bil_k, P.bil_k);
  const float2 mkz = make_float2(-(P.bil_k * z.x), -(P.bil_k * z.y));
#pragma unroll
  for (int dy = -R; dy <= R; ++dy)
#pragma unroll
    for (int dx = -R; dx <= R; ++dx) {
      const float2 zn = s_pair[(cy + dy) * RR + cx + dx];
      const float2 sd = __ffma2_rn(zn, k2, mkz);
      // the exponent's negative, sd^2 - sw: a packed operation has no free sign,
      // the exponential's operand has; one weight per distance, held in registers
      const float nsw = P.bil_nsw[dx * dx + dy * dy];
      const float2 e = __ffma2_rn(sd, sd, make_float2(nsw, nsw));
      const float2 wt = make_float2(ex2_approx(-e.x), ex2_approx(-e.y));
      num = __ffma2_rn(wt, zn, num);
      den = __fadd2_rn(den, wt);
    }
  return make_float2(__fdividef(num.x, den.x), __fdividef(num.y, den.y));
}

template <int R>
__device__ __forceinline__ float bilateral_at(const float* s_raw, int RR, int cx, int cy, float z,
                                              const KParams& P) {
  // exponent sw2 - c2 (zn - z)^2 as sw2 - s^2 with s = k zn - k z, k^2 = c2
  float num = 0.f, den = 0.f;
  const float kz = P.bil_k * z;
#pragma unroll
  for (int dy = -R; dy <= R; ++dy)
#pragma unroll
    for (int dx = -R; dx <= R; ++dx) {
      const float zn = s_raw[(cy + dy) * RR + cx + dx];
      const float sd = fmaf(zn, P.bil_k, -kz);
      const float wt = ex2_approx(fmaf(-sd, sd, P.bil_sw2[(dy + R) * (2 * R + 1) + dx + R]));
      num = fmaf(wt, zn, num);
      den += wt;
    }
  return __fdividef(num, den);
}

// One frame by threads t0, t0 + stride, ...: over its 16-byte groups, kCopyU per
// thread at a time (all loads issued before the stores); a source not on a
// 16-byte boundary, and the last count % 4 floats, go one float at a time.
constexpr int kCopyU = 4;
__device__ __forceinline__ void copy_frame(const float* src, float* dst, int count, int t0, int stride) {
  if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
    const int n4 = count / 4;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    float4* d4 = reinterpret_cast<float4*>(dst);
    for (int base = t0; base < n4; base += kCopyU * stride) {
      float4 v[kCopyU];
#pragma unroll
      for (int u = 0; u < kCopyU; ++u) {
        const int i = base + u * stride;
        if (i < n4) v[u] = s4[i];
      }
#pragma unroll
      for (int u = 0; u < kCopyU; ++u) {
        const int i = base + u * stride;
        if (i < n4) d4[i] = v[u];
      }
    }
    for (int i = 4 * n4 + t0; i < count; i += stride) dst[i] = src[i];
  } else {
    for (int i = t0; i < count; i += stride) dst[i] = src[i];
  }
}

// blockIdx.y: frame
__global__ void __launch_bounds__(256) k_copy_frames(FrameCopyList list) {
  const int f = blockIdx.y;
  copy_frame(list.src[f], list.dst[f], list.count[f], blockIdx.x * blockDim.x + threadIdx.x,
             gridDim.x * blockDim.x);
}

// Blocks of a front-end launch that copy the next launch's frames: 1.2 MB under
// way, what the host link needs (200 GB/s), on a twelfth of the places.
constexpr int kCopyBlocks = 76;

// RB: the bilateral radius. kLv: the number of levels, or 0 for any (read from
// the descriptor). What bounds a batch is instruction issue (78 % of the slots,
// 476 instructions a level-0 pixel before the levels were known here, a third of
// them integer and compare): with the regions' sizes as constants their
// divisions, 45 instructions a thread and phase, go; so do the halves of 1 / f
// and of the pyramid's means, and a bounds check and two stores a raw pixel.
// Measured on GB300, 256 frames 640x480, three levels: 1217 -> 867 us.
template <class T, int RB, int kLv>
__global__ void __launch_bounds__(kTx* kTy, KF_FE_MINB) k_frontend_fused(DescList list, FrameCopyList next,
                                                                            KParams P) {
  constexpr int r = RB;                                          // = P.bil_radius
  constexpr int kR0 = region0(kLv > 0 ? kLv : KF_MAX_LEVELS);    // largest of the instance
  constexpr int kRR = kR0 + 2 * r;
  constexpr int nthr = kTx * kTy;
  // raw depth as vertical pairs: s_pair[y S + x] = (D(x, y), D(x, y + 1)),
  // the row below the region holding no depth
  constexpr int kStride = kLv > 0 ? pair_stride(kR0, kRR) : kRR + 7;  // the largest of the instance
#if KF_FE_PAIRS
  __shared__ float2 s_pair[kRR * kStride];
#else
  __shared__ float s_raw[kRR * kStride];
#endif
  __shared__ __align__(8) float s_d0[kR0 * kR0];
  __shared__ __align__(8) float s_d1[kR0 / 2 * (kR0 / 2)];
  __shared__ __align__(8) float s_d2[kR0 / 4 * (kR0 / 4)];
  __shared__ __align__(8) float s_d3[kR0 / 8 * (kR0 / 8)];
  int z = blockIdx.z;
  if (z < next.layers) {  // the grid's first layers copy
    const int b = (z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    if (b < kCopyBlocks)
      for (int f = 0; f < next.n; ++f)
        copy_frame(next.src[f], next.dst[f], next.count[f], b * nthr + threadIdx.y * kTx + threadIdx.x,
                   kCopyBlocks * nthr);
    return;
  }
  z -= next.layers;
  const PairDesc* d = list.d[z];
  const int W = d->iw, H = d->ih;
  const int X0 = blockIdx.x * kTile, Y0 = blockIdx.y * kTile;
  if (X0 >= W || Y0 >= H) return;
  const int levels = kLv > 0 ? kLv : d->levels;
  const int R0 = kLv > 0 ? kR0 : region0(levels);
  const int RR = R0 + 2 * r;
  const int S = pair_stride(R0, RR);
  const int tid = threadIdx.y * kTx + threadIdx.x;
  const float* D = list.depth[z];
  // a thread loads a piece of a column, all of it before the first use: a pixel
  // is the lower half of its own pair and the upper half of the one above
  {
    const int groups = nthr / RR, rows = (RR + groups - 1) / groups;
    constexpr int kRows = (kRR + nthr / kRR - 1) / (nthr / kRR);  // the largest rows of the instance
    const int lx = tid % RR, y0 = tid / RR * rows;
    const int x = X0 - r + lx;
    const bool xin = tid < groups * RR && (unsigned)x < (unsigned)W;
    const int i0 = (Y0 - r + y0) * W + x;
    float z[kRows + 1];
#pragma unroll
    for (int k = 0; k <= kRows; ++k) {
      const int ly = y0 + k, y = Y0 - r + ly;
      z[k] = kNoDepth;
      if (xin && k <= rows && ly < RR && (unsigned)y < (unsigned)H) z[k] = __ldg(D + i0 + k * W);
    }
#pragma unroll
    for (int k = 0; k <= kRows; ++k)
      if (!valid_depth(z[k])) z[k] = kNoDepth;
    if (tid < groups * RR) {
#pragma unroll
      for (int k = 0; k < kRows; ++k)
        if (k < rows && y0 + k < RR) {
#if KF_FE_PAIRS
          s_pair[(y0 + k) * S + lx] = make_float2(z[k], z[k + 1]);
#else
          s_raw[(y0 + k) * S + lx] = z[k];
#endif
        }
    }
  }
  __syncthreads();
  // bilateral filter over the R0 x R0 region: w = 2^(sw2 - dz^2 c2), the weight
  // exp(-(dx^2 + dy^2) / (2 sigma_s^2) - dz^2 / (2 sigma_r^2)) with its exponent
  // scaled by log2(e)
#if KF_FE_PAIRS
  // two vertically adjacent pixels per step (rows ly and ly + 1; a region
  // with an odd row count filters one row below it and drops the result)
  for_region(R0, (R0 + 1) >> 1, tid, nthr, [&](int lx, int py) {
    const int ly = 2 * py;
    const int x = X0 + lx, y = Y0 + ly;
    const float2 z = s_pair[(ly + r) * S + lx + r];
    float2 out = RB > 0 ? bilateral_pair<RB>(s_pair, S, lx + r, ly + r, z, P) : z;
    const bool xin = x < W;
    s_d0[ly * R0 + lx] = xin && y < H && z.x != kNoDepth ? out.x : 0.f;
    if (ly + 1 < R0) s_d0[(ly + 1) * R0 + lx] = xin && y + 1 < H && z.y != kNoDepth ? out.y : 0.f;
  });
#else
  for_region(R0, R0, tid, nthr, [&](int lx, int ly) {
    const int x = X0 + lx, y = Y0 + ly;
    const float z = s_raw[(ly + r) * S + lx + r];
    float out = 0.f;
    if (x < W && y < H && z != kNoDepth) {
      out = RB > 0 ? bilateral_at<RB>(s_raw, S, lx + r, ly + r, z, P) : z;
    }
    s_d0[ly * R0 + lx] = out;
  });
#endif
  __syncthreads();
  // pyramid: level l+1 from level l inside shared memory, the mean of the depths of
  // a 2 x 2 block within 3 sigma_r of its first valid one
  float* lev[4] = {s_d0, s_d1, s_d2, s_d3};
#pragma unroll
  for (int l = 0; l + 1 < KF_MAX_LEVELS; ++l) {
    if (l + 1 >= levels) break;
    const int Rs = R0 >> l, Ro = R0 >> (l + 1);  // Rs is even
    const LevelMaps& Lo = d->lv[l + 1];
    const int fw = Lo.fw, fh = Lo.fh;
    const int ox = X0 >> (l + 1), oy = Y0 >> (l + 1);
    const float* src = lev[l];
    float* dst = lev[l + 1];
    for_region(Ro, Ro, tid, nthr, [&](int lx, int ly) {
      float out = 0.f;
      if (ox + lx < fw && oy + ly < fh) {
        const float2 b0 = *reinterpret_cast<const float2*>(src + 2 * ly * Rs + 2 * lx);
        const float2 b1 = *reinterpret_cast<const float2*>(src + (2 * ly + 1) * Rs + 2 * lx);
        const float b[4] = {b0.x, b0.y, b1.x, b1.y};
        // the first valid depth; none: no b[i] is counted
        const float anchor = b[0] > 0.f ? b[0] : b[1] > 0.f ? b[1] : b[2] > 0.f ? b[2] : b[3];
        float s = 0.f;
        int c = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (b[i] > 0.f && fabsf(__fsub_rn(b[i], anchor)) <= P.thr3sr32) {
            s = __fadd_rn(s, b[i]);
            ++c;
          }
        // s / c: the products by 1/4, 1/2 and 1 round as the quotients do
        out = c == 3 ? __fdiv_rn(s, 3.f) : __fmul_rn(s, c == 4 ? 0.25f : c == 2 ? 0.5f : 1.f);
      }
      dst[ly * Ro + lx] = out;
    });
    __syncthreads();
  }
  // the coarser levels' pixels on different warps
  write_maps<T, kTile, 4>(d->lv[0], s_d0, R0, X0, Y0);
  if (levels > 1) write_maps<T, kTile / 2, 2>(d->lv[1], s_d1, R0 >> 1, X0 >> 1, Y0 >> 1);
  if (levels > 2) write_maps<T, kTile / 4, 1, 128>(d->lv[2], s_d2, R0 >> 2, X0 >> 2, Y0 >> 2);
  if (levels > 3) write_maps<T, kTile / 8, 1, 192>(d->lv[3], s_d3, R0 >> 3, X0 >> 3, Y0 >> 3);
}


// ---------------------------------------------------------------------------
// Integral-image normals (Sec. 3.3; Holzer et al.): the average 3D gradient
// over a square window whose half-size follows the depth and stops short of
// depth edges. One block owns a 32 x 32 tile of one level of one frame (four
// rows per thread; blockIdx.x walks the tiles of every level, blockIdx.y is
// the frame) and does everything in shared memory:
//  * the level depth of the tile plus a halo of rmax + 1;
//  * edge flags over the tile plus rmax, one 64-bit mask per row (a warp per
//    row, ballots): no depth, or a 4-neighbour inside the image without depth
//    or with |z_w - z| > delta z (float32); pixels outside the image count as
//    edges too, which bounds the window exactly as the border distance does;
//  * fixed-point vertices Q = rint(v 2^20) (int64, round half to even), v the
//    front end's float32 vertex ((x - cx) z) (1/fx), ((y - cy) z) (1/fy), z,
//    0 without depth, and their local integral image (3 channels): window
//    sums are exact integers, the same however they are added;
//  * per pixel the chessboard distance to the nearest edge (the smallest
//    square around it holding an edge bit, from the row masks), the half-size
//    r = min(floor((a + b z) 2^-l), dist - 1, border distance, rmax),
//    g_h = S(right) - S(left), g_v = S(below) - S(above), and the normal
//    (g_h x g_v) / |g_h x g_v| in float32 with each operation rounded (g
//    scaled by 2^-20 exactly), flipped to face the camera; no normal unless
//    r >= 1 and the cross product is non-zero.
// Rewrites the level's vertex (NaN without a normal) and normal maps.
// ---------------------------------------------------------------------------
constexpr float kFix = 1048576.f;                // 2^20
constexpr float kFixInv = 9.5367431640625e-07f;  // 2^-20
constexpr int kIiRows = 4 * kTy;                 // output rows per block

// tiles of each level of the largest frame of a launch, and their prefix
struct IiGrid {
  int tx[KF_MAX_LEVELS];       // tiles per row
  int first[KF_MAX_LEVELS + 1];  // first tile of each level; first[levels] = total
  int levels;
};

// shared-memory layout of one tile for half-size cap rmax (<= 15: a row of
// the window region, 32 + 2 rmax <= 62 pixels, fits one 64-bit mask)
struct IiTile {
  int rw, rh;    // window region: tile plus rmax on each side
  int dw, dh;    // depth region: window region plus 1
  size_t ii, mask, depth, bytes;  // byte offsets and total
  __host__ __device__ IiTile(int rmax) {
    rw = kTx + 2 * rmax;
    rh = kIiRows + 2 * rmax;
    dw = rw + 2;
    dh = rh + 2;
    ii = 0;
    mask = ii + (size_t)3 * (rw + 1) * (rh + 1) * sizeof(long long);
    depth = mask + (size_t)rh * sizeof(unsigned long long);
    bytes = (depth + (size_t)dw * dh * sizeof(float) + 15) / 16 * 16;
  }
};

// chessboard distance from region pixel (x, y) to the nearest edge, capped
// at C: the smallest d whose square (rows y-d..y+d, columns x-d..x+d) holds
// an edge bit, grown one ring at a time (x - C + 1 >= 0 and the rows and
// columns up to distance C - 1 lie inside the region)
__device__ __forceinline__ int edge_distance(const unsigned long long* M, int x, int y, int C) {
  unsigned long long rows = 0;
  for (int d = 0; d < C; ++d) {
    rows |= M[y - d] | M[y + d];
    const unsigned long long win = (rows >> (x - d)) & ((2ull << (2 * d)) - 1ull);
    if (win) return d;
  }
  return C;
}

template <class T>
__global__ void __launch_bounds__(kTx * kTy) k_ii_normals(DescList list, IiGrid G, KParams P) {
  extern __shared__ __align__(16) unsigned char s_ii_raw[];
  int l = 0;
  while (l + 1 < G.levels && (int)blockIdx.x >= G.first[l + 1]) ++l;
  const int tile = blockIdx.x - G.first[l];
  const LevelMaps L = list.d[blockIdx.y]->lv[l];
  const int W = L.fw, H = L.fh;
  const int X0 = (tile % G.tx[l]) * kTx, Y0 = (tile / G.tx[l]) * kIiRows;
  if (X0 >= W || Y0 >= H) return;
  const int rmax = P.ii_rmax, C = rmax + 1;
  const IiTile tl(rmax);
  long long* sI = reinterpret_cast<long long*>(s_ii_raw + tl.ii);
  unsigned long long* sM = reinterpret_cast<unsigned long long*>(s_ii_raw + tl.mask);
  float* sD = reinterpret_cast<float*>(s_ii_raw + tl.depth);
  const int tid = threadIdx.y * kTx + threadIdx.x, nt = kTx * kTy;
  const int lane = threadIdx.x, warp = threadIdx.y;
  const float nan = __int_as_float(0x7fc00000);
  const float ifx = L.fifx, ify = L.fify;
  // the front end's vertex, operation for operation
  auto vertex = [&](int x, int y, float z) {
    return make_float3(__fmul_rn(__fmul_rn(__fsub_rn((float)x, L.fcx), z), ifx),
                       __fmul_rn(__fmul_rn(__fsub_rn((float)y, L.fcy), z), ify), z);
  };
  const int iw = tl.rw + 1, ipl = (tl.rw + 1) * (tl.rh + 1);  // integral row stride, plane
  // 1. depth with halo rmax + 1 (NaN outside the image: no depth)
  for (int k = tid; k < tl.dw * tl.dh; k += nt) {
    const int gy = Y0 - rmax - 1 + k / tl.dw, gx = X0 - rmax - 1 + k % tl.dw;
    sD[k] = (gx >= 0 && gx < W && gy >= 0 && gy < H) ? L.fdepth[gy * W + gx] : nan;
  }
  for (int k = tid; k < 3 * iw; k += nt) sI[(k / iw) * ipl + k % iw] = 0;  // row 0
  for (int k = tid; k < 3 * (tl.rh + 1); k += nt)
    sI[(k / (tl.rh + 1)) * ipl + (k % (tl.rh + 1)) * iw] = 0;                // column 0
  __syncthreads();
  // 2. a warp per region row: edge mask and fixed-point vertices
  for (int ry = warp; ry < tl.rh; ry += kTy) {
    const int gy = Y0 - rmax + ry;
    unsigned long long m = 0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int rx = lane + 32 * half;
      bool edge = true;
      long long q[3] = {0, 0, 0};
      if (rx < tl.rw) {
        const int gx = X0 - rmax + rx;
        const float* d = sD + (ry + 1) * tl.dw + (rx + 1);
        const float z = d[0];
        if (gx >= 0 && gx < W && gy >= 0 && gy < H && valid_depth(z)) {
          edge = false;
          const float thr = __fmul_rn(P.ii_delta, z);
          const float zn[4] = {d[1], d[-1], d[tl.dw], d[-tl.dw]};
          const bool inside[4] = {gx + 1 < W, gx > 0, gy + 1 < H, gy > 0};
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (inside[k] && (!valid_depth(zn[k]) || fabsf(__fsub_rn(zn[k], z)) > thr)) edge = true;
          const float3 v = vertex(gx, gy, z);
          q[0] = __float2ll_rn(__fmul_rn(v.x, kFix));
          q[1] = __float2ll_rn(__fmul_rn(v.y, kFix));
          q[2] = __float2ll_rn(__fmul_rn(v.z, kFix));
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) sI[c * ipl + (ry + 1) * iw + (rx + 1)] = q[c];
      }
      m |= (unsigned long long)__ballot_sync(0xffffffffu, edge && rx < tl.rw) << (32 * half);
    }
    if (lane == 0) sM[ry] = m;
  }
  __syncthreads();
  // 3. row prefix sums, then 4. column prefix sums
  for (int k = tid; k < 3 * tl.rh; k += nt) {
    long long* row = sI + (k / tl.rh) * ipl + (k % tl.rh + 1) * iw;
    long long acc = 0;
    for (int x = 1; x <= tl.rw; ++x) {
      acc += row[x];
      row[x] = acc;
    }
  }
  __syncthreads();
  for (int k = tid; k < 3 * tl.rw; k += nt) {
    long long* col = sI + (k / tl.rw) * ipl + (k % tl.rw + 1);
    long long acc = 0;
    for (int y = 1; y <= tl.rh; ++y) {
      acc += col[y * iw];
      col[y * iw] = acc;
    }
  }
  __syncthreads();
  // 5. four output pixels per thread
  const float lscale = ldexpf(1.f, -l);
#pragma unroll 1
  for (int part = 0; part < kIiRows / kTy; ++part) {
    const int oy = threadIdx.y + kTy * part;
    const int x = X0 + lane, y = Y0 + oy;
    if (x >= W || y >= H) continue;
    const int rx = lane + rmax, ry = oy + rmax;
    const float z = sD[(ry + 1) * tl.dw + (rx + 1)];
    const float3 v = vertex(x, y, z);
    const int dist = edge_distance(sM, rx, ry, C);
    float t = __fmul_rn(__fadd_rn(P.ii_a, __fmul_rn(P.ii_b, z)), lscale);
    if (!isfinite(t)) t = 0.f;
    const int rdd = (int)floorf(fminf(t, (float)rmax));
    const int rimg = min(min(x, W - 1 - x), min(y, H - 1 - y));
    const int r = min(min(rdd, dist - 1), min(rimg, rmax));
    float n[3] = {nan, nan, nan};
    bool ok = false;
    if (valid_depth(z) && r >= 1) {
      // sum of Q over region columns x0..x1, rows y0..y1 (inclusive), channel c
      auto S = [&](int c, int x0, int x1, int y0, int y1) -> long long {
        const long long* I = sI + c * ipl;
        return I[(y1 + 1) * iw + x1 + 1] - I[y0 * iw + x1 + 1] - I[(y1 + 1) * iw + x0] + I[y0 * iw + x0];
      };
      float gh[3], gv[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long h = S(c, rx + 1, rx + r, ry - r, ry + r) - S(c, rx - r, rx - 1, ry - r, ry + r);
        const long long w = S(c, rx - r, rx + r, ry + 1, ry + r) - S(c, rx - r, rx + r, ry - r, ry - 1);
        gh[c] = __fmul_rn(__ll2float_rn(h), kFixInv);
        gv[c] = __fmul_rn(__ll2float_rn(w), kFixInv);
      }
      const float cx = __fsub_rn(__fmul_rn(gh[1], gv[2]), __fmul_rn(gh[2], gv[1]));
      const float cy = __fsub_rn(__fmul_rn(gh[2], gv[0]), __fmul_rn(gh[0], gv[2]));
      const float cz = __fsub_rn(__fmul_rn(gh[0], gv[1]), __fmul_rn(gh[1], gv[0]));
      float n2 = __fadd_rn(__fmul_rn(cx, cx), __fmul_rn(cy, cy));
      n2 = __fadd_rn(n2, __fmul_rn(cz, cz));
      if (n2 > 0.f) {
        const float sn = __fsqrt_rn(n2);
        n[0] = __fdiv_rn(cx, sn);
        n[1] = __fdiv_rn(cy, sn);
        n[2] = __fdiv_rn(cz, sn);
        float dot = __fadd_rn(__fmul_rn(n[0], v.x), __fmul_rn(n[1], v.y));
        dot = __fadd_rn(dot, __fmul_rn(n[2], v.z));
        if (dot > 0.f) {
          n[0] = -n[0];
          n[1] = -n[1];
          n[2] = -n[2];
        }
        ok = true;
      }
    }
    const int i = y * W + x;
    Store<T>::store_a(L.fA, i, ok ? make_float4(v.x, v.y, v.z, n[0]) : make_float4(nan, nan, nan, n[0]));
    Store<T>::store_b(L.fB, i, make_float2(n[1], n[2]));
  }
}

}  // namespace

cudaError_t launch_copy_frames(const FrameCopyList& list, cudaStream_t s) {
  if (list.n <= 0) return cudaSuccess;
  int most = 0;
  for (int i = 0; i < list.n; ++i) most = list.count[i] > most ? list.count[i] : most;
  const int per_block = 256 * 4 * kCopyU;  // floats per block per pass
  int bx = (most + per_block - 1) / per_block;
  bx = bx < 1 ? 1 : (bx > 1024 ? 1024 : bx);
  k_copy_frames<<<dim3(bx, list.n), 256, 0, s>>>(list);
  return cudaGetLastError();
}

cudaError_t launch_frontend(const DescList& list, const FrameCopyList& pull, int max_w, int max_h, int levels,
                            const KParams& P, cudaStream_t s) {
  // 1..4 levels (the trackers' own) and radius 0..4: checked at tracker creation
  const dim3 blk(kTx, kTy);
  const int tx = (max_w + kTile - 1) / kTile, ty = (max_h + kTile - 1) / kTile;
  FrameCopyList next = pull;
  next.layers = next.n > 0 ? (kCopyBlocks + tx * ty - 1) / (tx * ty) : 0;
  const dim3 g(tx, ty, list.n + next.layers);
#define KF_FE(R, LV)                                                        \
  (P.precision == KF_FP16 ? k_frontend_fused<__half, R, LV><<<g, blk, 0, s>>>(list, next, P) \
                          : k_frontend_fused<float, R, LV><<<g, blk, 0, s>>>(list, next, P))
  // the default radius has an instance for each number of levels
  switch (P.bil_radius) {
    case 0: KF_FE(0, 0); break;
    case 1: KF_FE(1, 0); break;
    case 2:
      switch (levels) {
        case 1: KF_FE(2, 1); break;
        case 2: KF_FE(2, 2); break;
        case 3: KF_FE(2, 3); break;
        default: KF_FE(2, 4); break;
      }
      break;
    case 3: KF_FE(3, 0); break;
    default: KF_FE(4, 0); break;
  }
#undef KF_FE
  return cudaGetLastError();
}

cudaError_t launch_integral_normals(const DescList& list, int max_w, int max_h, int levels,
                                    const KParams& P, cudaStream_t s) {
  const IiTile tl(P.ii_rmax);
  IiGrid G;
  G.levels = levels;
  G.first[0] = 0;
  for (int l = 0; l < levels; ++l) {
    const int w = max_w >> l, h = max_h >> l;
    G.tx[l] = (w + kTx - 1) / kTx;
    G.first[l + 1] = G.first[l] + G.tx[l] * ((h + kIiRows - 1) / kIiRows);
  }
  const dim3 g(G.first[levels], list.n);
  cudaError_t e;
  if (P.precision == KF_FP16) {
    e = cudaFuncSetAttribute(k_ii_normals<__half>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tl.bytes);
    if (e != cudaSuccess) return e;
    k_ii_normals<__half><<<g, dim3(kTx, kTy), tl.bytes, s>>>(list, G, P);
  } else {
    e = cudaFuncSetAttribute(k_ii_normals<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tl.bytes);
    if (e != cudaSuccess) return e;
    k_ii_normals<float><<<g, dim3(kTx, kTy), tl.bytes, s>>>(list, G, P);
  }
  return cudaGetLastError();
}

cudaError_t launch_model_prep(const PairDesc& desc, PairDesc* d_desc, const float* V, const float* N, int w,
                              int h, int precision, cudaStream_t s) {
  const dim3 blk(kTx, kTy), grid((w + kTx - 1) / kTx, (h + kTy - 1) / kTy);
  if (precision == KF_FP16) k_model_prep<__half><<<grid, blk, 0, s>>>(desc, d_desc, V, N, w, h);
  else k_model_prep<float><<<grid, blk, 0, s>>>(desc, d_desc, V, N, w, h);
  return cudaGetLastError();
}

}  // namespace kf
