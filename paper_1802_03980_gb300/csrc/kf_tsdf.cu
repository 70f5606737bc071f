// Model producer: TSDF integration of depth frames into a cube of voxels and
// raycasting of the model's world vertex and normal maps (KinectFusion's
// mapping half; the paper keeps a 512^3 cube of at most 6 m side, Sec. 4.4,
// and aligns each frame to "the model reconstructed so far", Sec. 3).
//
// Every result that decides something discrete (the pixel a voxel projects
// to, the truncation test, the cell of a sample, a zero crossing) is an
// explicitly rounded float32 operation in a fixed order, so that a float32
// re-evaluation elsewhere reproduces the decisions bit for bit.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "kf_round.cuh"
#include "kf_internal.cuh"

namespace kf {
namespace {

struct VolGeom {
  int res;
  float s;           // voxel size: (float)side / (float)res
  float o[3];        // world position of the cube's lower corner
  float mu, w_max;
};

struct Cam32 {
  int w, h;
  float fx, fy, cx, cy;
};

__device__ __forceinline__ float rowv(const float* R, float t, float x, float y, float z) {
  float a = __fadd_rn(__fmul_rn(R[0], x), __fmul_rn(R[1], y));
  a = __fadd_rn(a, __fmul_rn(R[2], z));
  return __fadd_rn(a, t);
}

// world -> camera rows [R^T | -R^T t] (float32) for integration
struct Xf12 {
  float r[9];
  float t[3];
};

// Where the field may be observed and <= 0: a byte per brick (8^3 voxels), set
// for every brick that a cell with such a corner, or a cell one voxel beside
// it, is based in, and a byte per superbrick (8^3 bricks), set where one of its
// bricks is.
struct NearMap {
  unsigned char* brick;  // [nb^3]
  unsigned char* super;  // [ns^3]
  int nb, ns;
  // A warp marks for the values <= 0 it found in brick (bi, bj, bk);
  // low / high, per axis: non-zero where one lies within two voxels of the
  // brick's lower face / at its upper face (a cell is based one voxel below its
  // corners at most)
  __device__ __forceinline__ void mark(int bi, int bj, int bk, int lane, const unsigned (&low)[3],
                                       const unsigned (&high)[3]) const {
    if (lane >= 27) return;
    const int di = lane % 3 - 1, dj = lane / 3 % 3 - 1, dk = lane / 9 - 1;
    auto skip = [&](int d, int a) { return (d < 0 && !low[a]) || (d > 0 && !high[a]); };
    if (skip(di, 0) || skip(dj, 1) || skip(dk, 2)) return;
    const int i = bi + di, j = bj + dj, k = bk + dk;
    if ((unsigned)i >= (unsigned)nb || (unsigned)j >= (unsigned)nb || (unsigned)k >= (unsigned)nb) return;
    unsigned char* b = brick + ((size_t)k * nb + j) * nb + i;
    if (*b) return;
    *b = 1;
    super[((k >> 3) * ns + (j >> 3)) * ns + (i >> 3)] = 1;
  }
  // log2 of the edge in bricks of the aligned block around brick (i, j, k) that
  // holds nothing: 3, 0, or -1 where there may be something
  __device__ __forceinline__ int empty_block(int i, int j, int k) const {
    // outside the cube: a brick at a time up to its faces (half a voxel outside
    // the outermost cells)
    if ((unsigned)i >= (unsigned)nb || (unsigned)j >= (unsigned)nb || (unsigned)k >= (unsigned)nb) return 0;
    if (!__ldg(super + ((k >> 3) * ns + (j >> 3)) * ns + (i >> 3))) return 3;
    return __ldg(brick + ((unsigned)k * nb + j) * nb + i) ? -1 : 0;
  }
};

// a / b rounded to nearest, from y = 1 / b rounded to nearest: the quotient
// a y corrected by its exact remainder (Markstein, as rcp_rn_mid). No branch, and one
// reciprocal serves every division by b. For |b| in [2^-126, 2^126); a
// quotient too small or too large for the float32 range may differ from
// __fdiv_rn's in its last bits or come as NaN for an infinity, which no use
// here tells apart (a sum with a term of order one follows, or a range test).
__device__ __forceinline__ float div_rn_mid(float a, float b, float y) {
  const float q = __fmul_rn(a, y);
  return fmaf(fmaf(-q, b, a), y, q);
}

// A camera pixel's coordinate from (f p) / p_z + c: the nearest whole number,
// ties to even, as an integer outside [0, w) where it leaves the image. kAny:
// every input; otherwise w up to 2^22 and p_z of a middle exponent, y = 1 / p_z.
template <bool kAny>
__device__ __forceinline__ int pixel_of(float f, float p, float pz, float y, float c, int w) {
  const float a = __fmul_rn(f, p);
  if constexpr (kAny) {
    const float r = rintf(__fadd_rn(__fdiv_rn(a, pz), c));
    return r >= 0.f && r <= (float)(w - 1) ? (int)r : -1;
  } else {
    constexpr float kRint = 12582912.f;  // 1.5 2^23 (see project in kf_icp.cuh)
    return __float_as_int(__fadd_rn(__fadd_rn(div_rn_mid(a, pz, y), c), kRint)) - __float_as_int(kRint);
  }
}

// Integration visits only the voxels of bricks (8^3 voxels) that can lie in
// the image frustum: a brick is dropped when its bounding sphere lies wholly
// behind the camera or wholly outside one side plane of the frustum taken one
// pixel wider than the image on every side (so the float32 rounding of a
// voxel's projection, a small fraction of a pixel at depths >= 1 cm, cannot
// bring a dropped voxel into the image); bricks reaching closer than 1 cm to
// the camera plane are always kept. Every voxel that passes the per-voxel
// tests lies in a kept brick, so the volume is the same as from a pass over
// every voxel. Bricks wholly behind what the camera sees are dropped too: the
// depth image's largest valid depth over tiles of 16 x 16 pixels bounds the
// depths in the pixels the bounding sphere can project to, and a voxel farther
// than that depth plus mu is not updated.
constexpr int kBrick = 8;
constexpr int kDepthTile = 16;
// Tiles that a volume holds: frames up to 4096 x 4096 (larger ones are not tested
// against the depth). Allocated with it, since an integration allocates nothing
// for a device frame: it can be captured.
constexpr int kMaxTiles = 65536;
struct Frustum {
  float n[4][3];  // unit normals of the side planes (camera frame), inside: n . p >= 0
  float fx, fy, cx, cy;   // for the tiles (fx, fy > 0)
  int tw, th;             // tiles per row and column; 0: no depth test
};

// One warp per tile: its largest valid depth (0: none). The first thread also
// empties the brick list of the integration that follows.
__global__ void __launch_bounds__(256) k_depth_tiles(const float* D, int w, int h, int tw, int tiles,
                                                     float* tile_max, unsigned* count) {
  const int t = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (blockIdx.x == 0 && threadIdx.x == 0) *count = 0u;
  if (t >= tiles) return;
  const int x = (t % tw) * kDepthTile + (lane & 15), y0 = (t / tw) * kDepthTile + (lane >> 4);
  float m = 0.f;
#pragma unroll
  for (int k = 0; k < kDepthTile / 2; ++k) {
    const int y = y0 + 2 * k;
    if (x < w && y < h) {
      const float d = __ldg(D + (size_t)y * w + x);
      if (isfinite(d) && d > m) m = d;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) tile_max[t] = m;
}

__device__ __forceinline__ bool keep_brick(const VolGeom& g, const Xf12& xf, const Frustum& fr, int bi,
                                           int bj, int bk, const float* tile_max) {
  const float h = 0.5f * kBrick * g.s;  // half the brick's edge
  const float cx = g.o[0] + (float)(bi * kBrick) * g.s + h;
  const float cy = g.o[1] + (float)(bj * kBrick) * g.s + h;
  const float cz = g.o[2] + (float)(bk * kBrick) * g.s + h;
  const float px = xf.r[0] * cx + xf.r[1] * cy + xf.r[2] * cz + xf.t[0];
  const float py = xf.r[3] * cx + xf.r[4] * cy + xf.r[5] * cz + xf.t[1];
  const float pz = xf.r[6] * cx + xf.r[7] * cy + xf.r[8] * cz + xf.t[2];
  const float R = 1.7320509f * h + 1e-3f;  // bounding sphere plus a rounding margin
  if (pz < -R) return false;
  const float z0 = pz - R, z1 = pz + R;
  if (!(z0 >= 0.01f)) return true;
  for (int q = 0; q < 4; ++q)
    if (fr.n[q][0] * px + fr.n[q][1] * py + fr.n[q][2] * pz < -R) return false;
  if (fr.tw == 0) return true;
  // pixel bounds of the sphere's box, one pixel wider on every side
  const float i0 = 1.f / z0, i1 = 1.f / z1;
  const float ul = fr.fx * (px - R) * (px - R < 0.f ? i0 : i1) + fr.cx - 1.5f;
  const float uh = fr.fx * (px + R) * (px + R < 0.f ? i1 : i0) + fr.cx + 1.5f;
  const float vl = fr.fy * (py - R) * (py - R < 0.f ? i0 : i1) + fr.cy - 1.5f;
  const float vh = fr.fy * (py + R) * (py + R < 0.f ? i1 : i0) + fr.cy + 1.5f;
  constexpr float kInv = 1.f / kDepthTile;
  const int x0 = (int)fminf(fmaxf(ul * kInv, 0.f), (float)(fr.tw - 1));
  const int x1 = (int)fminf(fmaxf(uh * kInv, 0.f), (float)(fr.tw - 1));
  const int y0 = (int)fminf(fmaxf(vl * kInv, 0.f), (float)(fr.th - 1));
  const int y1 = (int)fminf(fmaxf(vh * kInv, 0.f), (float)(fr.th - 1));
  // a brick this close to the camera spans many tiles and is rarely hidden
  if ((x1 - x0 + 1) * (y1 - y0 + 1) > 128) return true;
  const float need = z0 - g.mu * 1.0001f - 1e-3f;
  for (int y = y0; y <= y1; ++y)
    for (int x = x0; x <= x1; ++x)
      if (__ldg(tile_max + y * fr.tw + x) >= need) return true;
  return false;
}

__global__ void __launch_bounds__(256) k_cull_bricks(VolGeom g, Xf12 xf, Frustum fr, int nb,
                                                     const float* tile_max, int* list, unsigned* count) {
  const int b = blockIdx.x * 256 + threadIdx.x;
  const int bi = b % nb, bj = (b / nb) % nb, bk = b / (nb * nb);
  const bool keep = bk < nb && keep_brick(g, xf, fr, bi, bj, bk, tile_max);
  // one atomic a warp
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  if (m == 0) return;
  const int lane = threadIdx.x & 31;
  unsigned base = 0;
  if (lane == 0) base = atomicAdd(count, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (keep) list[base + __popc(m & ((1u << lane) - 1u))] = b;
}

// Per voxel: F <- (W F + f) / (W + 1), W <- min(W + 1, w_max). 64 threads take
// a brick, each a column of eight voxels along z: the camera rows' x and y
// terms are formed once a column, and eight depth reads and eight voxels are in
// flight. What bounds it is issue (the projection and its tests) about as much
// as the 16 bytes a voxel; both divisions by p_z share one reciprocal, and free
// space (f = 1 on F = 1, or eta >= mu) takes no division. A brick that gets an
// observed value <= 0 marks itself and its neighbours in `near` (and their
// superbricks), where the raycast has to look; marks are never taken back
// (until a reset).
// Measured on GB300, 512^3 and 640x480, a whole call by events, calls in a row: 214
// us with a thread per voxel of every brick in the image, 57 to 70 us now (four
// scenes).
template <bool kAny>
__global__ void __launch_bounds__(256) k_integrate_bricks(float2* FW, VolGeom g, const float* D, Cam32 cam,
                                                          Xf12 xf, int nb, const int* list,
                                                          const unsigned* count, NearMap near) {
  const unsigned n = *count;
  const int sub = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int di = t % kBrick, dj = t / kBrick;
  const float rmu = kAny ? 0.f : __frcp_rn(g.mu);
  for (unsigned q = blockIdx.x * 4 + sub; q < n; q += gridDim.x * 4) {
    const int b = __ldg(list + q);
    const int bi = b % nb, bj = (b / nb) % nb, bk = b / (nb * nb);
    const int i = bi * kBrick + di, j = bj * kBrick + dj, k0 = bk * kBrick;
    const float fk0 = (float)k0;
    bool neg = false, neg_low = false, neg_high = false;
    if (i < g.res && j < g.res) {
      const float x = __fadd_rn(g.o[0], __fmul_rn((float)i + 0.5f, g.s));
      const float y = __fadd_rn(g.o[1], __fmul_rn((float)j + 0.5f, g.s));
      float xy[3];
#pragma unroll
      for (int r = 0; r < 3; ++r)
        xy[r] = __fadd_rn(__fmul_rn(xf.r[3 * r], x), __fmul_rn(xf.r[3 * r + 1], y));
      float d[kBrick], pz[kBrick];
#pragma unroll
      for (int k = 0; k < kBrick; ++k) {
        const float z = __fadd_rn(g.o[2], __fmul_rn(fk0 + (float)k + 0.5f, g.s));  // whole numbers: exact
        float p[3];  // rowv's order: ((R0 x + R1 y) + R2 z) + t
#pragma unroll
        for (int r = 0; r < 3; ++r)
          p[r] = __fadd_rn(__fadd_rn(xy[r], __fmul_rn(xf.r[3 * r + 2], z)), xf.t[r]);
        pz[k] = p[2];
        const float iz = kAny ? 0.f : rcp_rn_mid(p[2]);
        const int u = pixel_of<kAny>(cam.fx, p[0], p[2], iz, cam.cx, cam.w);
        const int v = pixel_of<kAny>(cam.fy, p[1], p[2], iz, cam.cy, cam.h);
        const bool in = p[2] > 0.f && (unsigned)u < (unsigned)cam.w && (unsigned)v < (unsigned)cam.h &&
                        k0 + k < g.res;
        if constexpr (kAny) d[k] = in ? __ldg(D + (size_t)v * cam.w + u) : 0.f;
        else d[k] = in ? __ldg(D + ((unsigned)v * cam.w + u)) : 0.f;
      }
      float2* col = FW + ((size_t)k0 * g.res + j) * g.res + i;
      const size_t plane = (size_t)g.res * g.res;
      bool use[kBrick];
      float2 fw[kBrick];
#pragma unroll
      for (int k = 0; k < kBrick; ++k) {
        use[k] = isfinite(d[k]) && d[k] > 0.f && __fsub_rn(d[k], pz[k]) >= -g.mu;
        if (use[k]) fw[k] = col[k * plane];
      }
#pragma unroll
      for (int k = 0; k < kBrick; ++k)
        if (use[k]) {
          const float eta = __fsub_rn(d[k], pz[k]);
          // eta / mu >= 1 where eta >= mu
          float f = 1.f;
          if (eta < g.mu) f = fminf(1.f, kAny ? __fdiv_rn(eta, g.mu) : div_rn_mid(eta, g.mu, rmu));
          const float w = fw[k].y, w1 = __fadd_rn(w, 1.f);
          // (w 1 + 1) / (w + 1) is 1
          float F = 1.f;
          if (f != 1.f || fw[k].x != 1.f) F = __fdiv_rn(__fadd_rn(__fmul_rn(w, fw[k].x), f), w1);
          col[k * plane] = make_float2(F, fminf(w1, g.w_max));
          if (F <= 0.f) {
            neg = true;
            if (k <= 1) neg_low = true;
            if (k == kBrick - 1) neg_high = true;
          }
        }
    }
    if (__any_sync(0xffffffffu, neg)) {
      auto some = [&](bool c) { return __ballot_sync(0xffffffffu, c); };
      const unsigned low[3] = {some(neg && di <= 1), some(neg && dj <= 1), some(neg_low)};
      const unsigned high[3] = {some(neg && di == kBrick - 1), some(neg && dj == kBrick - 1), some(neg_high)};
      near.mark(bi, bj, bk, threadIdx.x & 31, low, high);
    }
  }
}

__global__ void k_reset(float2* FW, size_t n) {
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n; v += (size_t)gridDim.x * blockDim.x)
    FW[v] = make_float2(1.f, 0.f);
}

// F and W of a run of voxels apart (inspection)
__global__ void k_split(const float2* FW, size_t n, float* F, float* W) {
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n; v += (size_t)gridDim.x * blockDim.x) {
    const float2 q = FW[v];
    F[v] = q.x;
    W[v] = q.y;
  }
}

// floor(x) as an integer, and as a float32 number in f; x outside +-2^22 (and
// NaN) gives an integer outside +-2^22. Additions instead of the conversion
// unit, which takes four times an addition's slot.
__device__ __forceinline__ int floor_of(float x, float& f) {
  constexpr float kMagic = 12582912.f;  // 1.5 2^23: its neighbours are whole numbers
  const float t = __fadd_rd(x, kMagic);
  f = __fsub_rn(t, kMagic);
  return __float_as_int(t) - __float_as_int(kMagic);
}
// a whole number within +-2^22 as float32
__device__ __forceinline__ float whole(int i) {
  constexpr float kMagic = 12582912.f;
  return __fsub_rn(__int_as_float(__float_as_int(kMagic) + i), kMagic);
}

// The eight corners around a world point: trilinear field value; false when the
// cell leaves the cube or has an unobserved corner (W = 0). Every load is
// issued before any is used. kAny: any voxel size; otherwise s in
// [2^-100, 2^100] and rs = 1 / s (see div_rn_mid).
template <bool kAny>
__device__ __forceinline__ bool sample(const float2* FW, const VolGeom& g, float rs, float qx, float qy,
                                       float qz, float& out) {
  auto grid = [&](float q, float o) {
    const float a = __fsub_rn(q, o);
    return __fsub_rn(kAny ? __fdiv_rn(a, g.s) : div_rn_mid(a, g.s, rs), 0.5f);
  };
  const float gx = grid(qx, g.o[0]), gy = grid(qy, g.o[1]), gz = grid(qz, g.o[2]);
  float fx0, fy0, fz0;
  const int x0 = floor_of(gx, fx0), y0 = floor_of(gy, fy0), z0 = floor_of(gz, fz0);
  const unsigned r = g.res, top = r - 1;  // the base lies in 0 .. res - 2
  if ((unsigned)x0 >= top || (unsigned)y0 >= top || (unsigned)z0 >= top) return false;
  const float tx = __fsub_rn(gx, fx0), ty = __fsub_rn(gy, fy0), tz = __fsub_rn(gz, fz0);
  const unsigned b0 = ((unsigned)z0 * r + y0) * r + x0, b1 = b0 + r * r;  // below 2^30
  const float2 c[8] = {__ldg(FW + b0),     __ldg(FW + b0 + 1),     __ldg(FW + (b0 + r)), __ldg(FW + (b0 + r) + 1),
                       __ldg(FW + b1),     __ldg(FW + b1 + 1),     __ldg(FW + (b1 + r)), __ldg(FW + (b1 + r) + 1)};
  const float w = fminf(fminf(fminf(c[0].y, c[1].y), fminf(c[2].y, c[3].y)),
                        fminf(fminf(c[4].y, c[5].y), fminf(c[6].y, c[7].y)));
  auto lerp = [](float a, float bb, float u) { return __fadd_rn(a, __fmul_rn(u, __fsub_rn(bb, a))); };
  const float c00 = lerp(c[0].x, c[1].x, tx), c10 = lerp(c[2].x, c[3].x, tx);
  const float c01 = lerp(c[4].x, c[5].x, tx), c11 = lerp(c[6].x, c[7].x, tx);
  out = lerp(lerp(c00, c10, ty), lerp(c01, c11, ty), tz);
  return w > 0.f;
}

struct RayParams {
  float R[9];   // camera -> world rotation (float32)
  float c[3];   // camera centre (world)
  float zn, zf, dz;
  int steps;    // samples k = 0 .. steps - 1 (z_k <= zf)
  float rs;     // 1 / voxel size
  int leap;     // empty bricks may be leapt over
};

// One thread per pixel: first front-to-back zero crossing of the field at the
// samples z_k = z_near + k dz.
//
// Only where an observed value <= 0 is near can a sample be <= 0 (a trilinear
// value of positive corners is positive, in float32 too), so a sample in a
// brick outside `near` is either unobserved or positive, and the ray leaps to
// the brick's (or superbrick's) far side; `near` covers cells one voxel beside
// the ones with such a corner, so the leaps' rounding does not matter.
// A leapt sample can only matter as the positive one before a crossing: it is
// then looked up. A ray whose last sample was negative does not leap (a
// positive one ends it).
// What bounds it is latency and issue per sample; a 640x480 view of a room takes
// about 115 samples a ray to the surface, of which this looks up a dozen.
// Measured on GB300, 512^3 and 640x480, calls in a row: 587 us looking up every
// sample, 78 to 88 us now (four scenes).
template <bool kAny>
__global__ void __launch_bounds__(128) k_raycast(const float2* FW, VolGeom g, NearMap near, Cam32 cam,
                                                 RayParams rp, float* V, float* N) {
  // a warp takes 8 x 4 pixels: its rays stay in the same bricks
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int u = blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7), v = blockIdx.y * 8 + (warp >> 1) * 4 + (lane >> 3);
  if (u >= cam.w || v >= cam.h) return;
  const float nan = __int_as_float(0x7fc00000);
  const float dcx = __fdiv_rn(__fsub_rn((float)u, cam.cx), cam.fx);
  const float dcy = __fdiv_rn(__fsub_rn((float)v, cam.cy), cam.fy);
  const float dx = rowv(rp.R + 0, 0.f, dcx, dcy, 1.f);
  const float dy = rowv(rp.R + 3, 0.f, dcx, dcy, 1.f);
  const float dzv = rowv(rp.R + 6, 0.f, dcx, dcy, 1.f);
  float out[6] = {nan, nan, nan, nan, nan, nan};
  auto depth_of = [&](int k) { return __fadd_rn(rp.zn, __fmul_rn((float)k, rp.dz)); };
  auto field = [&](float z, float& f) {
    return sample<kAny>(FW, g, rp.rs, __fadd_rn(rp.c[0], __fmul_rn(z, dx)), __fadd_rn(rp.c[1], __fmul_rn(z, dy)),
                        __fadd_rn(rp.c[2], __fmul_rn(z, dzv)), f);
  };
  // in bricks along each axis, per unit of camera depth (approximate: `near`
  // has a voxel's margin)
  const float per = rp.rs / (float)kBrick;
  const float bx0 = (rp.c[0] - g.o[0]) * per, by0 = (rp.c[1] - g.o[1]) * per, bz0 = (rp.c[2] - g.o[2]) * per;
  const float sx = dx * per, sy = dy * per, sz = dzv * per;
  const float ix = 1.f / sx, iy = 1.f / sy, iz = 1.f / sz, idz = 1.f / rp.dz;
  // the sample before k: known (have: observed, with value fp at depth zp) or leapt over
  bool known = true, have = false;
  float zp = 0.f, fp = 0.f;
  bool hit = false;
  float fh = 0.f;  // the value behind the surface
  for (int k = 0; k < rp.steps;) {
    const float z = depth_of(k);
    if (z > rp.zf) break;
    if (rp.leap && !(known && have && fp < 0.f)) {
      const float bx = bx0 + z * sx, by = by0 + z * sy, bz = bz0 + z * sz;
      float f;
      const int i = floor_of(bx, f), j = floor_of(by, f), l = floor_of(bz, f);
      const int size = near.empty_block(i, j, l);
      if (size >= 0) {
        // the depth at which the ray leaves the block (aligned, 1 << size bricks)
        const int low = ~0 << size;
        const float ex = whole((i & low) + (sx > 0.f ? 1 << size : 0));
        const float ey = whole((j & low) + (sy > 0.f ? 1 << size : 0));
        const float ez = whole((l & low) + (sz > 0.f ? 1 << size : 0));
        const float ze = fminf(fminf(sx != 0.f ? (ex - bx0) * ix : 3e38f, sy != 0.f ? (ey - by0) * iy : 3e38f),
                               sz != 0.f ? (ez - bz0) * iz : 3e38f);
        // samples up to here lie inside (less a margin for the rounding of ze and
        // of the quotient, below 1/50 of a sample up to 65536 samples)
        const float kn = fminf((ze - rp.zn) * idz, (float)rp.steps) - 0.05f;
        k = max(k + 1, (int)kn + 1);
        known = false;
        continue;
      }
    }
    float f;
    if (!field(z, f)) {
      known = true;
      have = false;
      ++k;
      continue;
    }
    if (f <= 0.f && !known) {
      zp = depth_of(k - 1);
      have = field(zp, fp);
      known = true;
    }
    if (known && have && fp > 0.f && f <= 0.f) {
      hit = true;
      fh = f;
      break;
    }
    if (known && have && fp < 0.f && f > 0.f) break;  // a back face: no surface
    known = have = true;
    zp = z;
    fp = f;
    ++k;
  }
  // the normals' samples once for all rays of the warp, wherever each met its
  // surface: inside the loop they ran for each sample at which some ray met it
  // (integration and raycast at 512^3 and 640x480, three volumes on three streams in
  // turn: 100 -> 96 us a pass)
  __syncwarp();
  if (hit) {
    const float zs = __fadd_rn(zp, __fmul_rn(rp.dz, __fdiv_rn(fp, __fsub_rn(fp, fh))));
    const float vx = __fadd_rn(rp.c[0], __fmul_rn(zs, dx));
    const float vy = __fadd_rn(rp.c[1], __fmul_rn(zs, dy));
    const float vz = __fadd_rn(rp.c[2], __fmul_rn(zs, dzv));
    float a[3], b[3];
    bool ok = sample<kAny>(FW, g, rp.rs, __fadd_rn(vx, g.s), vy, vz, a[0]);
    ok = sample<kAny>(FW, g, rp.rs, __fsub_rn(vx, g.s), vy, vz, b[0]) && ok;
    ok = sample<kAny>(FW, g, rp.rs, vx, __fadd_rn(vy, g.s), vz, a[1]) && ok;
    ok = sample<kAny>(FW, g, rp.rs, vx, __fsub_rn(vy, g.s), vz, b[1]) && ok;
    ok = sample<kAny>(FW, g, rp.rs, vx, vy, __fadd_rn(vz, g.s), a[2]) && ok;
    ok = sample<kAny>(FW, g, rp.rs, vx, vy, __fsub_rn(vz, g.s), b[2]) && ok;
    if (ok) {
      const float gx = a[0] - b[0], gy = a[1] - b[1], gz = a[2] - b[2];
      const float n2 = gx * gx + gy * gy + gz * gz;
      if (n2 > 0.f) {
        const float inv = 1.f / sqrtf(n2);
        out[0] = vx;
        out[1] = vy;
        out[2] = vz;
        out[3] = gx * inv;
        out[4] = gy * inv;
        out[5] = gz * inv;
      }
    }
  }
  const size_t p = ((size_t)v * cam.w + u) * 3;
  V[p] = out[0];
  V[p + 1] = out[1];
  V[p + 2] = out[2];
  N[p] = out[3];
  N[p + 1] = out[4];
  N[p + 2] = out[5];
}

}  // namespace
}  // namespace kf

using namespace kf;

struct kf_volume {
  kf_volume_params p;
  VolGeom g;
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float2* FW = nullptr;     // field and weight of each voxel
  NearMap near = {};
  float* tiles = nullptr;   // [kMaxTiles] largest depth per tile of the frame being integrated
  float* depth = nullptr;   // staging for host frames (grown on demand)
  size_t depth_cap = 0;
  float* maps = nullptr;    // staging for host outputs (grown on demand)
  size_t maps_cap = 0;
  int nb = 0;               // bricks per edge
  int* bricks = nullptr;    // kept bricks of the current integration (also what kf_volume_read takes apart)
  size_t bricks_cap = 0;    // ints
  unsigned* brick_count = nullptr;
  int sms = 1;
  std::string err;
};

namespace {

kf_status vfail(kf_volume* v, kf_status s, const std::string& msg) {
  if (v) v->err = msg;
  return s;
}

kf_status vcuda(kf_volume* v, cudaError_t e, const char* where) {
  if (v) v->err = std::string(where) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? KF_ERR_OOM : KF_ERR_CUDA;
}

#define KV_CK(v, expr)                                    \
  do {                                                    \
    cudaError_t e_ = (expr);                              \
    if (e_ != cudaSuccess) return vcuda(v, e_, #expr);    \
  } while (0)

bool cam_ok(const kf_intrinsics* K) {
  return K && K->width > 0 && K->height > 0 && std::isfinite(K->fx) && std::isfinite(K->fy) &&
         std::isfinite(K->cx) && std::isfinite(K->cy) && K->fx != 0.0 && K->fy != 0.0;
}

Cam32 cam32(const kf_intrinsics* K) {
  return Cam32{K->width, K->height, (float)K->fx, (float)K->fy, (float)K->cx, (float)K->cy};
}

bool pose_ok(const double* T) {
  if (!T) return false;
  for (int i = 0; i < 16; ++i)
    if (!std::isfinite(T[i])) return false;
  return true;
}

// a length whose reciprocal and quotients stay well inside the float32 range
bool mid_size(float a) { return a > 0x1p-60f && a < 0x1p60f; }

// Every voxel's camera depth is 0 or of a middle exponent: a sum of products of
// the pose's entries and voxel coordinates that are each 0 or not tiny, none
// of them large.
bool mid_lengths(const kf_volume* v, const Xf12& xf) {
  if (!(v->g.s > 0x1p-20f && v->g.s < 0x1p20f)) return false;
  auto mid = [](float a) { return a == 0.f || (std::fabs(a) > 0x1p-64f && std::fabs(a) < 0x1p40f); };
  for (int a = 0; a < 9; ++a)
    if (!mid(xf.r[a])) return false;
  for (int a = 0; a < 3; ++a)
    if (!mid(xf.t[a]) || !mid(v->g.o[a])) return false;
  return true;
}

kf_status grow(kf_volume* v, float** buf, size_t* cap, size_t bytes) {
  if (*cap >= bytes) return KF_OK;
  cudaFree(*buf);
  *buf = nullptr;
  *cap = 0;
  KV_CK(v, cudaMalloc(buf, bytes));
  *cap = bytes;
  return KF_OK;
}

}  // namespace

extern "C" {

kf_status kf_volume_default_params(kf_volume_params* p) {
  if (!p) return KF_ERR_INVALID_ARG;
  p->res = 512;
  p->side = 6.0f;
  p->origin[0] = -3.0f;
  p->origin[1] = -3.0f;
  p->origin[2] = -3.0f;
  p->mu = 0.05f;  // ~4 voxels: the band behind a surface must hold several samples
  p->w_max = 64.0f;
  return KF_OK;
}

kf_status kf_volume_create(const kf_volume_params* p, void* cuda_stream, kf_volume** out) {
  if (!p || !out) return KF_ERR_INVALID_ARG;
  *out = nullptr;
  if (p->res < 2 || p->res > 1024 || !(p->side > 0.f) || !std::isfinite(p->side) || !(p->mu > 0.f) ||
      !(p->w_max >= 1.f) || !std::isfinite(p->origin[0]) || !std::isfinite(p->origin[1]) ||
      !std::isfinite(p->origin[2]))
    return KF_ERR_INVALID_ARG;
  kf_volume* v = new (std::nothrow) kf_volume();
  if (!v) return KF_ERR_OOM;
  v->p = *p;
  v->g.res = p->res;
  v->g.s = p->side / (float)p->res;
  for (int a = 0; a < 3; ++a) v->g.o[a] = p->origin[a];
  v->g.mu = p->mu;
  v->g.w_max = p->w_max;
  cudaGetDevice(&v->device);
  cudaError_t e = cudaSuccess;
  if (cuda_stream) {
    v->stream = static_cast<cudaStream_t>(cuda_stream);
  } else {
    e = cudaStreamCreateWithFlags(&v->stream, cudaStreamNonBlocking);
    v->own_stream = e == cudaSuccess;
  }
  const size_t n = (size_t)p->res * p->res * p->res;
  v->nb = (p->res + kBrick - 1) / kBrick;
  if (e == cudaSuccess) e = cudaMalloc(&v->FW, n * sizeof(float2));
  v->near.nb = v->nb;
  v->near.ns = (v->nb + 7) / 8;
  const size_t nb3 = (size_t)v->nb * v->nb * v->nb, ns3 = (size_t)v->near.ns * v->near.ns * v->near.ns;
  if (e == cudaSuccess) e = cudaMalloc(&v->near.brick, nb3 + ns3);
  v->near.super = v->near.brick + nb3;
  v->bricks_cap = std::max(nb3, (size_t)1 << 16);
  if (e == cudaSuccess) e = cudaMalloc(&v->bricks, v->bricks_cap * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&v->tiles, kMaxTiles * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&v->brick_count, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&v->sms, cudaDevAttrMultiProcessorCount, v->device);
  if (e != cudaSuccess) {
    kf_volume_destroy(v);
    return e == cudaErrorMemoryAllocation ? KF_ERR_OOM : KF_ERR_CUDA;
  }
  const kf_status st = kf_volume_reset(v);
  if (st != KF_OK) {
    kf_volume_destroy(v);
    return st;
  }
  *out = v;
  return KF_OK;
}

void kf_volume_destroy(kf_volume* v) {
  if (!v) return;
  if (v->stream) cudaStreamSynchronize(v->stream);
  cudaFree(v->FW);
  cudaFree(v->near.brick);
  cudaFree(v->tiles);
  cudaFree(v->bricks);
  cudaFree(v->brick_count);
  cudaFree(v->depth);
  cudaFree(v->maps);
  if (v->own_stream) cudaStreamDestroy(v->stream);
  delete v;
}

const char* kf_volume_last_error(const kf_volume* v) { return v ? v->err.c_str() : "null volume"; }

kf_status kf_volume_reset(kf_volume* v) {
  if (!v) return KF_ERR_INVALID_ARG;
  const size_t n = (size_t)v->g.res * v->g.res * v->g.res;
  k_reset<<<1216, 256, 0, v->stream>>>(v->FW, n);
  KV_CK(v, cudaGetLastError());
  const size_t nb = v->near.nb, ns = v->near.ns;
  KV_CK(v, cudaMemsetAsync(v->near.brick, 0, nb * nb * nb + ns * ns * ns, v->stream));
  return KF_OK;
}

kf_status kf_volume_integrate(kf_volume* v, const float* depth, const kf_intrinsics* K,
                              const double pose[16], int is_device_ptr) {
  if (!v || !depth || !cam_ok(K) || !pose_ok(pose)) return vfail(v, KF_ERR_INVALID_ARG, "bad argument");
  const float* D = depth;
  if (!is_device_ptr) {
    const size_t bytes = (size_t)K->width * K->height * sizeof(float);
    kf_status st = grow(v, &v->depth, &v->depth_cap, bytes);
    if (st != KF_OK) return st;
    KV_CK(v, cudaMemcpyAsync(v->depth, depth, bytes, cudaMemcpyHostToDevice, v->stream));
    D = v->depth;
  }
  // rows of [R^T | -R^T t] in double, then rounded to float32
  Xf12 xf;
  for (int a = 0; a < 3; ++a) {
    double tt = 0.0;
    for (int b = 0; b < 3; ++b) {
      xf.r[a * 3 + b] = (float)pose[b * 4 + a];
      tt -= pose[b * 4 + a] * pose[b * 4 + 3];
    }
    xf.t[a] = (float)tt;
  }
  // side planes of the frustum one pixel wider than the image (u in
  // [-1.5, w + 0.5], v likewise); with a non-positive focal length nothing
  // is culled
  Frustum fr;
  memset(&fr, 0, sizeof(fr));
  if (K->fx > 0.0 && K->fy > 0.0) {
    const double nrm[4][3] = {{K->fx, 0.0, K->cx + 1.5},
                              {-K->fx, 0.0, K->width + 0.5 - K->cx},
                              {0.0, K->fy, K->cy + 1.5},
                              {0.0, -K->fy, K->height + 0.5 - K->cy}};
    for (int q = 0; q < 4; ++q) {
      const double l = std::sqrt(nrm[q][0] * nrm[q][0] + nrm[q][1] * nrm[q][1] + nrm[q][2] * nrm[q][2]);
      for (int a = 0; a < 3; ++a) fr.n[q][a] = (float)(nrm[q][a] / l);
    }
  }
  const int nb = v->nb;
  const int nbricks = nb * nb * nb;
  const int tw = (K->width + kDepthTile - 1) / kDepthTile, th = (K->height + kDepthTile - 1) / kDepthTile;
  // the projection in float32 pixels: images of sane size only
  const bool tiled = K->fx > 0.0 && K->fy > 0.0 && K->width <= 65536 && K->height <= 65536 && (long long)tw * th <= kMaxTiles;
  if (tiled) {
    fr.fx = (float)K->fx;
    fr.fy = (float)K->fy;
    fr.cx = (float)K->cx;
    fr.cy = (float)K->cy;
    fr.tw = tw;
    fr.th = th;
    k_depth_tiles<<<(tw * th + 7) / 8, 256, 0, v->stream>>>(D, K->width, K->height, tw, tw * th, v->tiles,
                                                            v->brick_count);
    KV_CK(v, cudaGetLastError());
  } else {
    KV_CK(v, cudaMemsetAsync(v->brick_count, 0, sizeof(unsigned), v->stream));
  }
  k_cull_bricks<<<(nbricks + 255) / 256, 256, 0, v->stream>>>(v->g, xf, fr, nb, v->tiles, v->bricks,
                                                              v->brick_count);
  KV_CK(v, cudaGetLastError());
  // the short forms of the divisions and roundings hold for images up to 2^22
  // pixels wide and lengths of everyday exponents
  const bool any = K->width > (1 << 22) || K->height > (1 << 22) || (long long)K->width * K->height > 0x7fffffffLL ||
                    !mid_size(v->g.mu) || !mid_lengths(v, xf);
  auto kernel = any ? k_integrate_bricks<true> : k_integrate_bricks<false>;
  kernel<<<v->sms * 8, 256, 0, v->stream>>>(v->FW, v->g, D, cam32(K), xf, nb, v->bricks, v->brick_count, v->near);
  KV_CK(v, cudaGetLastError());
  if (!is_device_ptr) KV_CK(v, cudaStreamSynchronize(v->stream));
  return KF_OK;
}

kf_status kf_volume_raycast(kf_volume* v, const kf_intrinsics* K, const double pose[16],
                            float z_near, float z_far, float dz, float* vertex, float* normal,
                            int is_device_ptr) {
  if (!v || !cam_ok(K) || !pose_ok(pose) || !vertex || !normal || !(dz > 0.f) ||
      !(z_far >= z_near) || !std::isfinite(z_near) || !std::isfinite(z_far))
    return vfail(v, KF_ERR_INVALID_ARG, "bad argument");
  const double nsteps = std::floor(((double)z_far - (double)z_near) / (double)dz) + 2.0;
  if (nsteps > 1e6) return vfail(v, KF_ERR_INVALID_ARG, "more than 1e6 samples per ray");
  RayParams rp;
  for (int a = 0; a < 3; ++a) {
    for (int b = 0; b < 3; ++b) rp.R[a * 3 + b] = (float)pose[a * 4 + b];
    rp.c[a] = (float)pose[a * 4 + 3];
  }
  rp.zn = z_near;
  rp.zf = z_far;
  rp.dz = dz;
  rp.steps = (int)nsteps;  // the kernel also stops once z_k > z_far
  const size_t px = (size_t)K->width * K->height;
  float* Vd = vertex;
  float* Nd = normal;
  if (!is_device_ptr) {
    kf_status st = grow(v, &v->maps, &v->maps_cap, px * 6 * sizeof(float));
    if (st != KF_OK) return st;
    Vd = v->maps;
    Nd = v->maps + px * 3;
  }
  rp.rs = 1.f / v->g.s;
  // leaps are measured in float32 bricks: everyday lengths only
  rp.leap = mid_size(v->g.s) && mid_size(dz) && rp.steps <= 65536 && std::fabs(z_near) < 0x1p60f &&
            std::fabs(z_far) < 0x1p60f;
  for (int a = 0; a < 3; ++a)
    if (!(std::fabs(rp.c[a]) < 0x1p20f * v->g.s && std::fabs(v->g.o[a]) < 0x1p20f * v->g.s)) rp.leap = 0;
  // a leap's block lies within 2^22 bricks of the cube
  const double reach = std::max(std::fabs((double)z_near), std::fabs((double)z_far)) *
                       (1.0 + (K->width + std::fabs(K->cx)) / std::fabs(K->fx) + (K->height + std::fabs(K->cy)) / std::fabs(K->fy));
  if (!(reach < 0x1p22 * v->g.s)) rp.leap = 0;
  const dim3 grid((K->width + 15) / 16, (K->height + 7) / 8);
  auto kernel = mid_size(v->g.s) ? k_raycast<false> : k_raycast<true>;
  kernel<<<grid, 128, 0, v->stream>>>(v->FW, v->g, v->near, cam32(K), rp, Vd, Nd);
  KV_CK(v, cudaGetLastError());
  if (!is_device_ptr) {
    KV_CK(v, cudaMemcpyAsync(vertex, Vd, px * 3 * sizeof(float), cudaMemcpyDeviceToHost, v->stream));
    KV_CK(v, cudaMemcpyAsync(normal, Nd, px * 3 * sizeof(float), cudaMemcpyDeviceToHost, v->stream));
    KV_CK(v, cudaStreamSynchronize(v->stream));
  }
  return KF_OK;
}

kf_status kf_volume_read(kf_volume* v, float* F, float* W) {
  if (!v) return KF_ERR_INVALID_ARG;
  const size_t n = (size_t)v->g.res * v->g.res * v->g.res;
  KV_CK(v, cudaStreamSynchronize(v->stream));
  // a part of the volume at a time, taken apart in the brick list (the stream is idle)
  const size_t most = v->bricks_cap / 2;
  float* part = reinterpret_cast<float*>(v->bricks);
  for (size_t at = 0; at < n; at += most) {
    const size_t m = std::min(most, n - at);
    k_split<<<1216, 256, 0, v->stream>>>(v->FW + at, m, part, part + most);
    KV_CK(v, cudaGetLastError());
    KV_CK(v, cudaStreamSynchronize(v->stream));
    if (F) KV_CK(v, cudaMemcpy(F + at, part, m * sizeof(float), cudaMemcpyDeviceToHost));
    if (W) KV_CK(v, cudaMemcpy(W + at, part + most, m * sizeof(float), cudaMemcpyDeviceToHost));
  }
  return KF_OK;
}

}  // extern "C"
