// Ray kernels of the HRT hot path on sm_103a: the KDK step with the A/B recursion and readout (Alg. 1),
// the force-free drift, and the binning of the convergence power spectrum.
//
// One thread per ray.  The line-of-sight node table of the step (FP64 on the host, rounded to float32 here)
// travels in the kernel parameters, so every warp reads it by broadcast from the constant bank.  The ray
// angle stays FP64; per half shell the FP64 base position r_ref * theta is split into an integer cell and a
// float32 fraction, and each node adds a small float32 offset (r_j - r_ref) theta, so the float32
// interpolation position keeps ~1e-6-cell accuracy at any distance from the observer.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.h"
#include "mesh_kernels.h"
#include "packed.cuh"
#include "ray_position.cuh"
#include "readout.cuh"

namespace hrt {

struct HalfKick {
  float kx, ky;              // kick
  float j00, j01, j10, j11;  // dK/dtheta
};

__device__ __forceinline__ void base_position(const RayStepParams& p, double obs, double r_ref, double theta, int& i0,
                                              float& f0) {
  if (p.theta32) {
    const int n = p.n;
    const double cell = p.cell;
    // the FP32 ablation: the position and its cell split in single precision
    float uf = (static_cast<float>(obs) + static_cast<float>(r_ref) * static_cast<float>(theta)) / static_cast<float>(cell);
    uf -= static_cast<float>(n) * floorf(uf / static_cast<float>(n));
    const float flf = floorf(uf);
    i0 = static_cast<int>(flf);
    if (i0 >= n) i0 -= n;
    if (i0 < 0) i0 += n;
    f0 = uf - flf;
    return;
  }
  split_cell(p, line_of_sight_cell(p, obs, r_ref, theta), i0, f0);
}

// Wraps k into [0, n): one compare for the usual k within a box of [0, n), the division only beyond.
__device__ __forceinline__ int wrap_cell(int k, int n) {
  if (k >= n) {
    k -= n;
    if (k >= n) k %= n;
  } else if (k < 0) {
    k += n;
    if (k < 0) {
      k %= n;
      if (k < 0) k += n;
    }
  }
  return k;
}

__device__ __forceinline__ void node_axis(int i0, float f0, float off, int n, int& i, float& f) {
  float u = f0 + off;
  float fl = floorf(u);
  f = u - fl;
  i = wrap_cell(i0 + static_cast<int>(fl), n);
}

__device__ __forceinline__ HalfKick half_kick(const RayStepParams& p, int j0, int j1, double th_x, double th_y,
                                              double ref_r, const float* __restrict__ gx,
                                              const float* __restrict__ gy) {
  HalfKick h{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (j1 <= j0) return h;
  const int n = p.n;
  int bx, by;
  float fbx, fby;
  base_position(p, p.obs_x, ref_r, th_x, bx, fbx);
  base_position(p, p.obs_y, ref_r, th_y, by, fby);
  const float tx = static_cast<float>(th_x), ty = static_cast<float>(th_y);
  const int64_t nn = n;
  for (int j = j0; j < j1; ++j) {
    const float dr = p.dr[j];
    int ix, iy;
    float fx, fy;
    node_axis(bx, fbx, dr * tx, n, ix, fx);
    node_axis(by, fby, dr * ty, n, iy, fy);
    const int iz = p.kz[j];
    const int jz = iz + 1 == n ? 0 : iz + 1;
    const float fz = p.fz[j];
    const int jx = ix + 1 == n ? 0 : ix + 1, jy = iy + 1 == n ? 0 : iy + 1;
    const int64_t r00 = (ix * nn + iy) * nn, r01 = (ix * nn + jy) * nn, r10 = (jx * nn + iy) * nn,
                  r11 = (jx * nn + jy) * nn;
    // z-interpolated columns of both fields
    float ax00 = __ldg(gx + r00 + iz), ax01 = __ldg(gx + r01 + iz), ax10 = __ldg(gx + r10 + iz),
          ax11 = __ldg(gx + r11 + iz);
    float bx00 = __ldg(gx + r00 + jz), bx01 = __ldg(gx + r01 + jz), bx10 = __ldg(gx + r10 + jz),
          bx11 = __ldg(gx + r11 + jz);
    float ay00 = __ldg(gy + r00 + iz), ay01 = __ldg(gy + r01 + iz), ay10 = __ldg(gy + r10 + iz),
          ay11 = __ldg(gy + r11 + iz);
    float by00 = __ldg(gy + r00 + jz), by01 = __ldg(gy + r01 + jz), by10 = __ldg(gy + r10 + jz),
          by11 = __ldg(gy + r11 + jz);
    float x00 = ax00 + fz * (bx00 - ax00), x01 = ax01 + fz * (bx01 - ax01);
    float x10 = ax10 + fz * (bx10 - ax10), x11 = ax11 + fz * (bx11 - ax11);
    float y00 = ay00 + fz * (by00 - ay00), y01 = ay01 + fz * (by01 - ay01);
    float y10 = ay10 + fz * (by10 - ay10), y11 = ay11 + fz * (by11 - ay11);
    // bilinear value and transverse derivatives (per cell; 1/cell is folded into cwr)
    float vx0 = x00 + fy * (x01 - x00), vx1 = x10 + fy * (x11 - x10);
    float vy0 = y00 + fy * (y01 - y00), vy1 = y10 + fy * (y11 - y10);
    float vx = vx0 + fx * (vx1 - vx0), vy = vy0 + fx * (vy1 - vy0);
    float dxx = vx1 - vx0, dyx = vy1 - vy0;
    float dxy = (x01 - x00) + fx * ((x11 - x10) - (x01 - x00));
    float dyy = (y01 - y00) + fx * ((y11 - y10) - (y01 - y00));
    const float c = p.cw[j], cr = p.cwr[j];
    h.kx += c * vx;
    h.ky += c * vy;
    h.j00 += cr * dxx;
    h.j01 += cr * dxy;
    h.j10 += cr * dyx;
    h.j11 += cr * dyy;
  }
  return h;
}

// ---- node planes --------------------------------------------------------------------------------------------
// Every ray meets node j at the same z, so the z-interpolation of the two fields at (x, y) is the same for all rays of
// that cell: 78 of them at 2048^2 rays over 10 degrees and 1024^3 cells.  plane_kernel makes it once per cell of the
// rays' bounding box into planes [node][y][x] of (d_x phi, d_y phi), 26 MB in that step (60 nodes); the ray kernel then
// gathers four 8-byte corners per node, x fastest as a warp's 16 neighbouring pixels lie, instead of sixteen floats from
// sixteen columns, with the same arithmetic on the same numbers.  At 2048^2 rays, 60 nodes and 1024^3 cells a step takes
// 0.60 ms (bounds 21, planes 21, rays 551 us) against 1.57 ms, at 512^2 rays and 256^3 cells 0.12 against 0.31 ms.
//
// Most bytes of a step's planes.  A step whose box needs more, or holds more cells than there are rays, has chosen its kernel
// by then (the box is known on the device only) and gathers from the fields at four blocks per SM, 2 to 20 % slower than
// with no planes asked for; so the limit lies beyond the steps of a long run.  The planes need not stay in L2: a tile of
// rays reads a few cells of each.  Steps 48 and 64 of the 2048^2-ray reverse run (1024^3 cells, 85 and 98 nodes, 120 and 334 MB
// of planes): 0.87 and 1.31 ms, fields 2.42 and 4.91, and 2.79 and 5.05 while the limit was 96 MB.  It is in proportion
// to the rays because the workspace is as large, and mapping it costs the first step of a context 1.5 us per MB (and
// again whenever the nodes of a step become more): with 512 MB for all, 0.4 ms of an 8.2 ms run with 512^2 rays.  (Above one
// cell per ray the planes would still pay: 256^2 rays, 64 nodes, 2.2 cells per ray 77 and 268 us, 7.3 cells 176 and 266.)
constexpr size_t kPlaneBytesPerRay = 384, kPlaneBytesLow = size_t{96} << 20, kPlaneBytes = size_t{512} << 20;

// The box comes from the rays' largest and smallest angles, found on the device in the same step (ray_bounds_kernel).  It
// is in unwrapped cells and may be wider than the mesh, so that the ray kernel wraps nothing; a ray that leaves it (the
// angles of the second half shell have moved) reads the fields themselves.
struct PlaneBox {
  int x0, y0, rx, ry;  // first cell and extent per axis; rx = 0: no planes in this step
};

struct RayPlanes {
  // workspace: ordered keys of max theta_x, max -theta_x, max theta_y, max -theta_y; blocks done; the box
  unsigned long long* key;
  unsigned* done;
  PlaneBox* box;
  float2* data;
  int64_t capacity;   // of data, in pairs
  double r_lo, r_hi;  // smallest and largest node radius
};

// The bits of a double as an unsigned key of the same order, above 0 for every number; and of its negative.
__device__ __forceinline__ unsigned long long order_key(unsigned long long b) { return b >> 63 ? ~b : b | (1ull << 63); }
__device__ __forceinline__ double from_order_key(unsigned long long k) {
  return __longlong_as_double(static_cast<long long>(k >> 63 ? k ^ (1ull << 63) : ~k));
}

// Two cells to spare on either side, and the upper corner's.  Extent 0 where that is no sensible number of cells.
__device__ __forceinline__ void plane_axis(double obs, double t_lo, double t_hi, const RayPlanes& q, double cell, int& first,
                                           int& extent) {
  const double a = fmin(q.r_lo * t_lo, q.r_hi * t_lo), b = fmax(q.r_lo * t_hi, q.r_hi * t_hi);
  const double lo = floor((obs + a) / cell) - 2.0, size = floor((obs + b) / cell) + 4.0 - lo;
  const bool fine = size >= 1.0 && size <= 65536.0 && fabs(lo) < 1e9;
  extent = fine ? static_cast<int>(size) : 0;
  first = fine ? static_cast<int>(lo) : 0;
}

// Bounds of all angles; the last block to end makes the box of them.  Integer work only per ray: this part has few FP64 lanes.
__global__ void __launch_bounds__(256) ray_bounds_kernel(const ulonglong2* __restrict__ theta, int64_t nr,
                                                         const __grid_constant__ RayStepParams p, RayPlanes q) {
  unsigned long long k[4] = {0, 0, 0, 0};
  for (int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; r < nr;
       r += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const ulonglong2 t = theta[r];
    k[0] = max(k[0], order_key(t.x));
    k[1] = max(k[1], order_key(t.x ^ (1ull << 63)));
    k[2] = max(k[2], order_key(t.y));
    k[3] = max(k[3], order_key(t.y ^ (1ull << 63)));
  }
  __shared__ unsigned long long best[4];
  if (threadIdx.x < 4) best[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long other = __shfl_xor_sync(0xffffffffu, k[i], o);
      k[i] = max(k[i], other);
    }
    if ((threadIdx.x & 31) == 0) atomicMax(best + i, k[i]);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int i = 0; i < 4; ++i) atomicMax(q.key + i, best[i]);
  __threadfence();
  if (atomicAdd(q.done, 1u) + 1u != gridDim.x) return;
  __threadfence();
  unsigned long long all[4];
  for (int i = 0; i < 4; ++i) all[i] = atomicMax(q.key + i, 0ull);
  PlaneBox b;
  plane_axis(p.obs_x, -from_order_key(all[1]), from_order_key(all[0]), q, p.cell, b.x0, b.rx);
  plane_axis(p.obs_y, -from_order_key(all[3]), from_order_key(all[2]), q, p.cell, b.y0, b.ry);
  // fewer rays than cells, or too much to hold: the gather of each ray is the cheaper way
  const int64_t cells = static_cast<int64_t>(b.rx) * b.ry;
  if (cells > nr || cells * (p.n1 + p.n2) > q.capacity || b.ry == 0) b.rx = 0;
  *q.box = b;
}

// A block makes 32 nodes' planes of 8 x 8 cells: a lane per node, so that a warp reads the columns' z runs as they lie (a
// thread per cell walking up its column read 32 bytes at a time from rows far apart: 111 us instead of 21 for 60 nodes of 232 x 232
// cells), eight
// cells of independent loads per warp, and the planes' rows leave through shared memory.
constexpr int kPlaneNodes = 32, kPlaneSide = 8;

__global__ void __launch_bounds__(256) plane_kernel(const float* __restrict__ gx, const float* __restrict__ gy,
                                                    const __grid_constant__ RayStepParams p, RayPlanes q) {
  __shared__ float2 tile[kPlaneSide * kPlaneSide][kPlaneNodes + 1];
  const PlaneBox b = *q.box;
  if (b.rx == 0) return;
  const int nodes = p.n1 + p.n2, chunks = (nodes + kPlaneNodes - 1) / kPlaneNodes;
  const int tiles_x = (b.rx + kPlaneSide - 1) / kPlaneSide, tiles_y = (b.ry + kPlaneSide - 1) / kPlaneSide;
  const int n = p.n, total = tiles_x * tiles_y * chunks, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t plane = static_cast<int64_t>(b.ry) * b.rx;
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const int t = w / chunks, j0 = (w - t * chunks) * kPlaneNodes, ty = t / tiles_x;
    const int x0 = (t - ty * tiles_x) * kPlaneSide, y0 = ty * kPlaneSide;
    const int j = min(j0 + lane, nodes - 1), iz = p.kz[j], jz = iz + 1 == n ? 0 : iz + 1;
    const float fz = p.fz[j];
    int cx = (b.x0 + x0 + warp) % n;
    if (cx < 0) cx += n;
    float ax[kPlaneSide], ay[kPlaneSide], ux[kPlaneSide], uy[kPlaneSide];
#pragma unroll
    for (int y = 0; y < kPlaneSide; ++y) {  // cells past the box: read, not written
      int cy = (b.y0 + y0 + y) % n;
      if (cy < 0) cy += n;
      const int64_t col = (static_cast<int64_t>(cx) * n + cy) * n;
      ax[y] = __ldg(gx + col + iz);
      ay[y] = __ldg(gy + col + iz);
      ux[y] = __ldg(gx + col + jz);
      uy[y] = __ldg(gy + col + jz);
    }
#pragma unroll
    for (int y = 0; y < kPlaneSide; ++y)
      tile[y * kPlaneSide + warp][lane] = make_float2(ax[y] + fz * (ux[y] - ax[y]), ay[y] + fz * (uy[y] - ay[y]));
    __syncthreads();
    const int xs = min(kPlaneSide, b.rx - x0), ys = min(kPlaneSide, b.ry - y0), count = min(kPlaneNodes, nodes - j0);
    for (int k = threadIdx.x; k < count * kPlaneSide * kPlaneSide; k += blockDim.x) {
      const int x = k % kPlaneSide, y = k / kPlaneSide % kPlaneSide, i = k / (kPlaneSide * kPlaneSide);
      if (x < xs && y < ys)
        q.data[(j0 + i) * plane + static_cast<int64_t>(y0 + y) * b.rx + x0 + x] = tile[y * kPlaneSide + x][i];
    }
    __syncthreads();
  }
}

// half_kick on the planes of nodes j0 .. j1; node[j] = (dr, cw, cwr).  The nodes' cells lie between those of the first and
// the last, so that one look decides for all of them.
__device__ __forceinline__ HalfKick half_kick_planes(const RayStepParams& p, int j0, int j1, double th_x, double th_y,
                                                     double ref_r, double fixed_r, const float* __restrict__ gx,
                                                     const float* __restrict__ gy, const float2* __restrict__ planes,
                                                     const float4* __restrict__ node, const PlaneBox& b) {
  if (j1 <= j0) return HalfKick{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  // cell and fraction from one 32.32 fixed-point number per axis (2^-32 cells; a float's fraction has 2^-24): a single FP64
  // FMA and a conversion, with the step's constants scaled on the host
  const long long kx = __double2ll_rd(fma(fixed_r, th_x, p.fixed_obs_x)), ky = __double2ll_rd(fma(fixed_r, th_y, p.fixed_obs_y));
  const int cx = static_cast<int>(kx >> 32), cy = static_cast<int>(ky >> 32);
  const float fbx = static_cast<float>(static_cast<unsigned>(kx)) * 0x1p-32f, fby = static_cast<float>(static_cast<unsigned>(ky)) * 0x1p-32f;
  // Cells within 2^29 of the origin, looked at before anything is compared with them: the box starts within 1e9, so that no
  // sum of cells leaves int.  Angles that are not finite, or out of the conversion's range, saturate and end outside.
  constexpr unsigned kCells = 1u << 29;
  const bool near = static_cast<unsigned>(cx) + kCells < 2 * kCells && static_cast<unsigned>(cy) + kCells < 2 * kCells;
  const int bx = static_cast<int>(static_cast<unsigned>(cx) - static_cast<unsigned>(b.x0)),
            by = static_cast<int>(static_cast<unsigned>(cy) - static_cast<unsigned>(b.y0));
  const float tx = static_cast<float>(th_x), ty = static_cast<float>(th_y);
  auto inside = [&](float dr) {
    const float px = fbx + dr * tx, py = fby + dr * ty;
    if (!(fabsf(px) < 65536.f && fabsf(py) < 65536.f)) return false;
    const int x = bx + static_cast<int>(floorf(px)), y = by + static_cast<int>(floorf(py));
    return x >= 0 && x + 1 < b.rx && y >= 0 && y + 1 < b.ry;
  };
  if (!near || !inside(node[j0].x) || !inside(node[j1 - 1].x))
    return half_kick(p, j0, j1, th_x, th_y, ref_r, gx, gy);
  // floor as an integer from the bits of floor + 1.5 2^23 (the conversion unit is slow); the offset of those bits is taken
  // off here once
  constexpr float kMagic = 12582912.f;
  constexpr unsigned kMagicBits = 0x4b400000u;
  const int plane = b.rx * b.ry;
  const unsigned offset = static_cast<unsigned>(by) * static_cast<unsigned>(b.rx) + static_cast<unsigned>(bx) -
                          kMagicBits * static_cast<unsigned>(b.rx + 1);
  const float2* __restrict__ at = planes + static_cast<int64_t>(j0) * plane;
  // both components of a corner, (d_x phi, d_y phi), side by side
  u64 k = 0, jx = 0, jy = 0;
  auto corner = [](const float2* c) { return static_cast<u64>(__ldg(reinterpret_cast<const unsigned long long*>(c))); };
#pragma unroll 4
  for (int j = j0; j < j1; ++j, at += plane) {
    const float4 nd = node[j];
    const float px = fbx + nd.x * tx, py = fby + nd.x * ty;
    const float lx = floorf(px), ly = floorf(py);
    const u64 fx = both(px - lx), fy = both(py - ly);
    const unsigned e = offset + static_cast<unsigned>(__float_as_int(ly + kMagic)) * static_cast<unsigned>(b.rx) +
                       static_cast<unsigned>(__float_as_int(lx + kMagic));
    const float2* __restrict__ q = at + static_cast<int>(e);
    const u64 c0 = corner(q), c2 = corner(q + 1), c1 = corner(q + b.rx), c3 = corner(q + b.rx + 1);
    // bilinear value and transverse derivatives (per cell; 1/cell is folded into cwr)
    const u64 e0 = sub2(c1, c0), e1 = sub2(c3, c2);
    const u64 v0 = fma2(fy, e0, c0), v1 = fma2(fy, e1, c2), dx = sub2(v1, v0);
    const u64 v = fma2(fx, dx, v0), dy = fma2(fx, sub2(e1, e0), e0);
    const u64 cw = both(nd.y), cr = both(nd.z);
    k = fma2(cw, v, k);
    jx = fma2(cr, dx, jx);
    jy = fma2(cr, dy, jy);
  }
  const float2 kk = unpack(k), jxx = unpack(jx), jyy = unpack(jy);
  return {kk.x, kk.y, jxx.x, jyy.x, jxx.y, jyy.y};
}

// Cell and fraction on a box axis of a sky coordinate (cell i_s, fraction f_s) under sign sgn and a translation
// of sh cells: u -> sgn u + sh (mod n); a flipped point on a cell face stays on the face (lower cell).
__device__ __forceinline__ void box_axis(int i_s, float f_s, int sgn, int sh, int n, int& ib, float& fb) {
  if (sgn > 0) {
    ib = i_s + sh;
    fb = f_s;
  } else if (f_s > 0.f) {
    ib = sh - i_s - 1;
    fb = 1.f - f_s;
  } else {
    ib = sh - i_s;
    fb = 0.f;
  }
  ib = wrap_cell(ib, n);
}

__device__ __forceinline__ int pick(int axis, int a, int b, int c) { return axis == 0 ? a : (axis == 1 ? b : c); }
__device__ __forceinline__ float pickf(int axis, float a, float b, float c) { return axis == 0 ? a : (axis == 1 ? b : c); }

// Trilinear value of field f at box cell (ix, iy, iz) + (fx, fy, fz) and its derivatives (per cell) along
// the three box axes.
__device__ __forceinline__ void trilinear3(const float* __restrict__ f, int64_t r00, int64_t r01, int64_t r10,
                                           int64_t r11, int iz, int jz, float fx, float fy, float fz, float& v,
                                           float& dX, float& dY, float& dZ) {
  const float a00 = __ldg(f + r00 + iz), a01 = __ldg(f + r01 + iz), a10 = __ldg(f + r10 + iz), a11 = __ldg(f + r11 + iz);
  const float z00 = __ldg(f + r00 + jz) - a00, z01 = __ldg(f + r01 + jz) - a01, z10 = __ldg(f + r10 + jz) - a10,
              z11 = __ldg(f + r11 + jz) - a11;
  const float e00 = a00 + fz * z00, e01 = a01 + fz * z01, e10 = a10 + fz * z10, e11 = a11 + fz * z11;
  const float h0 = e01 - e00, h1 = e11 - e10;
  const float g0 = e00 + fy * h0, g1 = e10 + fy * h1;
  v = g0 + fx * (g1 - g0);
  dX = g1 - g0;
  dY = h0 + fx * (h1 - h0);
  const float q0 = z00 + fy * (z01 - z00), q1 = z10 + fy * (z11 - z10);
  dZ = q0 + fx * (q1 - q0);
}

// Half kick through a light cone tiled by rotated and translated replicas: each node is mapped into its
// replica's box frame; the sky gradient component a is sign_a times field perm_a there, and its derivative along
// sky axis b is sign_a sign_b times the box derivative along perm_b.
__device__ __forceinline__ HalfKick half_kick_tiled(const RayStepParams& p, int j0, int j1, double th_x, double th_y,
                                                    double ref_r, const float* __restrict__ gx,
                                                    const float* __restrict__ gy, const float* __restrict__ gz) {
  HalfKick h{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (j1 <= j0) return h;
  const int n = p.n;
  int bx, by;
  float fbx, fby;
  base_position(p, p.obs_x, ref_r, th_x, bx, fbx);
  base_position(p, p.obs_y, ref_r, th_y, by, fby);
  const float tx = static_cast<float>(th_x), ty = static_cast<float>(th_y);
  const int64_t nn = n;
  for (int j = j0; j < j1; ++j) {
    const float dr = p.dr[j];
    int ix, iy;
    float fx, fy;
    node_axis(bx, fbx, dr * tx, n, ix, fx);
    node_axis(by, fby, dr * ty, n, iy, fy);
    const int R = p.rep[j];
    const int p0 = p.rperm[R][0], p1 = p.rperm[R][1];
    const int s0 = p.rsign[R][0], s1 = p.rsign[R][1];
    int c0, c1;
    float q0, q1;
    box_axis(ix, fx, s0, p.rshift[R][0], n, c0, q0);
    box_axis(iy, fy, s1, p.rshift[R][1], n, c1, q1);
    const int c2 = p.kz[j];
    const float q2 = p.fz[j];
    // box-frame cell and fraction per box axis (axis p0 from sky x, p1 from sky y, the other from the line of sight)
    const int jx_ = pick(0 == p0 ? 0 : (0 == p1 ? 1 : 2), c0, c1, c2), jy_ = pick(1 == p0 ? 0 : (1 == p1 ? 1 : 2), c0, c1, c2),
              jz_ = pick(2 == p0 ? 0 : (2 == p1 ? 1 : 2), c0, c1, c2);
    const float gfx = pickf(0 == p0 ? 0 : (0 == p1 ? 1 : 2), q0, q1, q2), gfy = pickf(1 == p0 ? 0 : (1 == p1 ? 1 : 2), q0, q1, q2),
                gfz = pickf(2 == p0 ? 0 : (2 == p1 ? 1 : 2), q0, q1, q2);
    const int kx = jx_ + 1 == n ? 0 : jx_ + 1, ky = jy_ + 1 == n ? 0 : jy_ + 1, kz2 = jz_ + 1 == n ? 0 : jz_ + 1;
    const int64_t r00 = (jx_ * nn + jy_) * nn, r01 = (jx_ * nn + ky) * nn, r10 = (kx * nn + jy_) * nn,
                  r11 = (kx * nn + ky) * nn;
    const float* fa = p0 == 0 ? gx : (p0 == 1 ? gy : gz);
    const float* fb = p1 == 0 ? gx : (p1 == 1 ? gy : gz);
    float va, aX, aY, aZ, vb, bX, bY, bZ;
    trilinear3(fa, r00, r01, r10, r11, jz_, kz2, gfx, gfy, gfz, va, aX, aY, aZ);
    trilinear3(fb, r00, r01, r10, r11, jz_, kz2, gfx, gfy, gfz, vb, bX, bY, bZ);
    const float ss = static_cast<float>(s0 * s1);
    const float c = p.cw[j], cr = p.cwr[j];
    h.kx += c * (s0 * va);
    h.ky += c * (s1 * vb);
    h.j00 += cr * pickf(p0, aX, aY, aZ);
    h.j01 += cr * (ss * pickf(p1, aX, aY, aZ));
    h.j10 += cr * (ss * pickf(p0, bX, bY, bZ));
    h.j11 += cr * pickf(p1, bX, bY, bZ);
  }
  return h;
}

// One thread per ray.  On the planes the loop is bound by the latency and the issue of its gathers, four 8-byte loads a
// node: four blocks of 128 per SM (128 registers) and four nodes in flight measured 551 us at 2048^2 rays and 60 nodes,
// against 643 us with five blocks, 601 us with two nodes in flight, 684 us with eight.  From the fields
// __launch_bounds__(128, 1) leaves the register count to the compiler (72): 1.05 ms per step against 1.29 ms with 56.
enum class Gather { kFields, kTiled, kPlanes };

template <Gather G>
__global__ void __launch_bounds__(128, G == Gather::kPlanes ? 4 : 1) ray_step_kernel(double2* __restrict__ theta, float2* __restrict__ eta,
                                                       float4* __restrict__ Amat, float4* __restrict__ Bmat,
                                                       int64_t nr, const float* __restrict__ gx,
                                                       const float* __restrict__ gy, const __grid_constant__ RayStepParams p,
                                                       float* __restrict__ maps, const float* __restrict__ gz,
                                                       RayPlanes planes) {
  constexpr bool TILED = G == Gather::kTiled;
  extern __shared__ float4 node[];  // planes: (dr, cw, cwr) of the nodes
  PlaneBox box{0, 0, 0, 0};
  if constexpr (G == Gather::kPlanes) {
    box = *planes.box;
    for (int j = threadIdx.x; j < p.n1 + p.n2; j += blockDim.x) node[j] = make_float4(p.dr[j], p.cw[j], p.cwr[j], 0.f);
    __syncthreads();
  }
  auto half = [&](int j0, int j1, const double2& t, double ref_r) {
    if constexpr (TILED) return half_kick_tiled(p, j0, j1, t.x, t.y, ref_r, gx, gy, gz);
    if constexpr (G == Gather::kPlanes)
      if (box.rx > 0) return half_kick_planes(p, j0, j1, t.x, t.y, ref_r, p.fixed_r[j0 > 0], gx, gy, planes.data, node, box);
    return half_kick(p, j0, j1, t.x, t.y, ref_r, gx, gy);
  };
  int64_t r;
  if (p.tile_w > 0) {
    // 16 x 8 pixel tiles in row-major tile order; a warp covers 16 x 2 neighbouring pixels
    const unsigned tiles_x = static_cast<unsigned>(p.tile_w) >> 4;
    const unsigned tx = blockIdx.x % tiles_x, ty = blockIdx.x / tiles_x;
    const int64_t x = tx * 16 + (threadIdx.x & 15), y = ty * 8 + (threadIdx.x >> 4);
    r = y * p.tile_w + x;
  } else {
    r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  }
  if (r >= nr) return;
  double2 th = theta[r];
  float2 et = eta[r];
  float4 A = Amat[r], B = Bmat[r];

  HalfKick h = half(0, p.n1, th, p.ref_r[0]);
  et.x += h.kx;
  et.y += h.ky;
  // B += J A (row-major 2x2: x = 11, y = 12, z = 21, w = 22)
  B.x += h.j00 * A.x + h.j01 * A.z;
  B.y += h.j00 * A.y + h.j01 * A.w;
  B.z += h.j10 * A.x + h.j11 * A.z;
  B.w += h.j10 * A.y + h.j11 * A.w;
  // drift: theta in FP64, A in float32
  const double d = p.drift_d;
  if (p.theta32) {
    const float df = static_cast<float>(d);
    th.x = static_cast<double>(static_cast<float>(th.x) + df * et.x);
    th.y = static_cast<double>(static_cast<float>(th.y) + df * et.y);
  } else {
    th.x += d * static_cast<double>(et.x);
    th.y += d * static_cast<double>(et.y);
  }
  A.x += p.drift * B.x;
  A.y += p.drift * B.y;
  A.z += p.drift * B.z;
  A.w += p.drift * B.w;
  h = half(p.n1, p.n1 + p.n2, th, p.ref_r[1]);
  et.x += h.kx;
  et.y += h.ky;
  B.x += h.j00 * A.x + h.j01 * A.z;
  B.y += h.j00 * A.y + h.j01 * A.w;
  B.z += h.j10 * A.x + h.j11 * A.z;
  B.w += h.j10 * A.y + h.j11 * A.w;

  theta[r] = th;
  eta[r] = et;
  Amat[r] = A;
  Bmat[r] = B;
  if (maps != nullptr) {
    float k, g1, g2, om;
    readout(A, k, g1, g2, om);
    if (p.map_accumulate) {
      // O = sum_n n_g(chi_n) O_n (Eq. obs_accum): this step's observables with the caller's weight
      const float w = p.map_weight;
      maps[r] += w * k;
      maps[r + nr] += w * g1;
      maps[r + 2 * nr] += w * g2;
      maps[r + 3 * nr] += w * om;
    } else {
      maps[r] = k;
      maps[r + nr] = g1;
      maps[r + 2 * nr] = g2;
      maps[r + 3 * nr] = om;
    }
  }
}

// Workspace of planes: stream-ordered from a pool of the library's own, which keeps at most kPlanePoolBytes per
// device between calls (given back by ray_planes_release): a ray step's largest, and a ray-mesh slab beside it.
constexpr size_t kPlanePoolBytes = kPlaneBytes + (size_t{64} << 20);
constexpr int kPoolDevices = 16;
static std::mutex g_plane_mutex;
static cudaMemPool_t g_plane_pool[kPoolDevices] = {};

static cudaMemPool_t plane_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= kPoolDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_plane_mutex);
  if (!g_plane_pool[dev]) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    uint64_t keep = kPlanePoolBytes;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    g_plane_pool[dev] = pool;
  }
  return g_plane_pool[dev];
}

void ray_planes_release() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= kPoolDevices) return;
  std::lock_guard<std::mutex> lock(g_plane_mutex);
  if (g_plane_pool[dev]) cudaMemPoolTrimTo(g_plane_pool[dev], 0);
}

void* plane_workspace(size_t bytes, cudaStream_t s) {
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return nullptr;
  }
  if (inject_alloc_failure()) return nullptr;
  cudaMemPool_t pool = plane_pool();
  void* work = nullptr;
  if (pool && cudaMallocFromPoolAsync(&work, bytes, pool, s) == cudaSuccess) return work;
  cudaGetLastError();
  return nullptr;
}

// Rays, and rays times nodes, from which the three small launches before the step's (about 12 us) pay, at any shape above:
// planes and fields at the line, 256^3 cells: 128^2 rays and 256 nodes 60 and 129 us, 256^2 and 64 38 and 63 us, 512^2 and 16
// 45 and 53 us; below it 256^2 and 16 30 and 29 us, 128^2 and 32 29 and 25 us.
constexpr int64_t kPlaneRays = 1 << 14, kPlaneWork = 1 << 22;

hrt_status launch_ray_step(const hrt_rays& rays, const float* gx, const float* gy, const RayStepParams& p,
                           float* maps, cudaStream_t s, const float* gz) {
  if (rays.n_rays == 0) return HRT_OK;
  if (p.tiled && !gz) return fail(HRT_ERR_INVALID_ARG, "light-cone tiling needs the third gradient component");
  auto* kernel = p.tiled ? ray_step_kernel<Gather::kTiled> : ray_step_kernel<Gather::kFields>;
  RayPlanes q{};
  const int nodes = p.n1 + p.n2;
  char* work = nullptr;
  if (!p.tiled && !p.theta32 && rays.n_rays >= kPlaneRays && rays.n_rays * nodes >= kPlaneWork) {
    // a step without the workspace gathers from the fields
    const size_t most = static_cast<size_t>(nodes) * rays.n_rays * sizeof(float2);  // no more cells than rays
    const size_t bytes = std::min(most, std::clamp(kPlaneBytesPerRay * rays.n_rays, kPlaneBytesLow, kPlaneBytes));
    work = static_cast<char*>(plane_workspace(256 + bytes, s));
    if (work) {
      q.key = reinterpret_cast<unsigned long long*>(work);
      q.done = reinterpret_cast<unsigned*>(work + 32);
      q.box = reinterpret_cast<PlaneBox*>(work + 48);
      q.data = reinterpret_cast<float2*>(work + 256);
      q.capacity = static_cast<int64_t>(bytes / sizeof(float2));
      q.r_lo = p.r_lo;
      q.r_hi = p.r_hi;
      kernel = ray_step_kernel<Gather::kPlanes>;
    }
  }
  if (work) {
    const cudaError_t cleared = cudaMemsetAsync(work, 0, 256, s);
    if (cleared != cudaSuccess) {
      cudaFreeAsync(work, s);
      return cuda_status(cleared, "workspace of the ray planes");
    }
    ray_bounds_kernel<<<std::min(blocks_for(rays.n_rays, 256), 152u * 8u), 256, 0, s>>>(
        reinterpret_cast<const ulonglong2*>(rays.theta), rays.n_rays, p, q);
    plane_kernel<<<152 * 8, 256, 0, s>>>(gx, gy, p, q);
  }
  kernel<<<blocks_for(rays.n_rays, 128), 128, work ? nodes * sizeof(float4) : 0, s>>>(
      reinterpret_cast<double2*>(rays.theta), reinterpret_cast<float2*>(rays.eta),
      reinterpret_cast<float4*>(rays.A), reinterpret_cast<float4*>(rays.B), rays.n_rays, gx, gy, p, maps, gz, q);
  count_launches(work ? 3 : 1);
  const cudaError_t launched = cudaGetLastError();
  if (work) cudaFreeAsync(work, s);
  return cuda_status(launched, "ray_step_kernel");
}

__global__ void ray_drift_kernel(double2* __restrict__ theta, const float2* __restrict__ eta,
                                 float4* __restrict__ Amat, const float4* __restrict__ Bmat, int64_t nr, double d) {
  int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (r >= nr) return;
  double2 th = theta[r];
  float2 et = eta[r];
  th.x += d * static_cast<double>(et.x);
  th.y += d * static_cast<double>(et.y);
  theta[r] = th;
  float4 A = Amat[r];
  const float4 B = Bmat[r];
  const float df = static_cast<float>(d);
  A.x += df * B.x;
  A.y += df * B.y;
  A.z += df * B.z;
  A.w += df * B.w;
  Amat[r] = A;
}

hrt_status launch_ray_drift_free(const hrt_rays& rays, double d, cudaStream_t s) {
  if (rays.n_rays == 0) return HRT_OK;
  ray_drift_kernel<<<blocks_for(rays.n_rays, 256), 256, 0, s>>>(
      reinterpret_cast<double2*>(rays.theta), reinterpret_cast<const float2*>(rays.eta),
      reinterpret_cast<float4*>(rays.A), reinterpret_cast<const float4*>(rays.B), rays.n_rays, d);
  HRT_LAUNCHED("ray_drift_kernel");
  return HRT_OK;
}

__global__ void ray_readout_kernel(const float4* __restrict__ Amat, int64_t nr, float* __restrict__ maps) {
  int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (r >= nr) return;
  float k, g1, g2, om;
  readout(Amat[r], k, g1, g2, om);
  maps[r] = k;
  maps[r + nr] = g1;
  maps[r + 2 * nr] = g2;
  maps[r + 3 * nr] = om;
}

hrt_status launch_ray_readout(const hrt_rays& rays, float* maps, cudaStream_t s) {
  if (rays.n_rays == 0) return HRT_OK;
  ray_readout_kernel<<<blocks_for(rays.n_rays, 256), 256, 0, s>>>(reinterpret_cast<const float4*>(rays.A),
                                                                  rays.n_rays, maps);
  HRT_LAUNCHED("ray_readout_kernel");
  return HRT_OK;
}

// theta0 may be theta itself (initialisation in place)
__global__ void rays_init_kernel(double2* theta, float2* __restrict__ eta, float4* __restrict__ Amat,
                                 float4* __restrict__ Bmat, const double2* theta0, int64_t nr) {
  int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (r >= nr) return;
  theta[r] = theta0[r];
  eta[r] = make_float2(0.f, 0.f);
  Amat[r] = make_float4(1.f, 0.f, 0.f, 1.f);
  Bmat[r] = make_float4(0.f, 0.f, 0.f, 0.f);
}

hrt_status launch_rays_init(const hrt_rays& rays, const double* theta0, cudaStream_t s) {
  if (rays.n_rays == 0) return HRT_OK;
  rays_init_kernel<<<blocks_for(rays.n_rays, 256), 256, 0, s>>>(
      reinterpret_cast<double2*>(rays.theta), reinterpret_cast<float2*>(rays.eta),
      reinterpret_cast<float4*>(rays.A), reinterpret_cast<float4*>(rays.B),
      reinterpret_cast<const double2*>(theta0), rays.n_rays);
  HRT_LAUNCHED("rays_init_kernel");
  return HRT_OK;
}

// ---------------------------------------------------------------------------------------------------------
// Power-spectrum binning of the m x (m/2+1) half spectrum of kappa.  Column kz = 1..m/2-1 stands for two
// modes (n and -n); kz = 0 and kz = m/2 for one.  The bin rule of the header is increasing in |n|^2, an integer, so the
// host finds each bin's first |n|^2 with it (FP64) and the kernel compares integers.
//
// Bound by latency and the few FP64 lanes of this part: an FP64 logarithm and square root and three FP64 shared-memory
// atomics per mode, most lanes of a warp on the same bin, took 880 us at m = 2048.  A warp now takes 256 columns of
// the rows nx and -nx, whose geometry is the same; a lane's modes climb through the bins, so it adds in registers, and
// what lanes hold goes to shared memory, summed over the warp, where a bin ends and at the end: 70 us with a shared-memory
// atomic per lane there, 34 us with the sum.  A lane's sums of |n| and of the squares are three floats each, which round less
// than FP64; they become FP64 when they leave the lane.  (With two floats each P was off by up to 4.6e-15 from the sums
// of the same spectrum in 80 bits, with FP64 by 1.2e-15, now by 0.7e-15; a call takes the same time with two and three.)
// ---------------------------------------------------------------------------------------------------------
constexpr int kBinColumns = 256;

// Whether x^2, its rounding error and sums of a warp's many stay within float's normal range (0 does; NaN does not).
__device__ __forceinline__ bool moderate(float x) { return x == 0.f || (fabsf(x) > 1e-12f && fabsf(x) < 1e15f); }
__device__ __forceinline__ bool moderate(float2 z) { return moderate(z.x) && moderate(z.y); }

// A sum in three floats of falling size: what a float sum rounds away goes to the next, so that 2^-70 of it is lost at
// most, less than in FP64.
struct Sum3 {
  float hi, mid, lo;
};
__device__ __forceinline__ float two_sum(float a, float b, float& rounded) {
  const float s = __fadd_rn(a, b), back = __fsub_rn(s, a);
  rounded = __fadd_rn(__fsub_rn(a, __fsub_rn(s, back)), __fsub_rn(b, back));
  return s;
}
// x to the middle of the sum: a rounding error of what went on top
__device__ __forceinline__ void add_small(Sum3& s, float x) {
  float e;
  s.mid = two_sum(s.mid, x, e);
  s.lo += e;
}
__device__ __forceinline__ void add_to(Sum3& s, float x) {
  float e;
  s.hi = two_sum(s.hi, x, e);
  add_small(s, e);
}
__device__ __forceinline__ double value(const Sum3& s) { return static_cast<double>(s.hi) + (static_cast<double>(s.mid) + s.lo); }

// s += scale x^2; scale a power of two.
__device__ __forceinline__ void add_square(Sum3& s, float x, float scale) {
  const float sx = scale * x, q = __fmul_rn(sx, x);
  add_to(s, q);
  add_small(s, __fmaf_rn(sx, x, -q));
}

// s += modes sqrt(n2); modes a power of two, n2 > 0.  The float root, then the residual's share of it to first order as
// a quotient with its own residual, and the second order: 2^-70.
__device__ __forceinline__ void add_root(Sum3& s, int n2, int modes) {
  const float a = static_cast<float>(n2), root = sqrtf(a), twice = 2.f * root;
  float left;
  const float r = two_sum(__fmaf_rn(-root, root, a), static_cast<float>(n2 - static_cast<int>(a)), left);
  const float c = r / twice, rest = (__fmaf_rn(-twice, c, r) + left - c * c) / twice;
  add_to(s, root * modes);
  add_small(s, c * modes);
  s.lo += rest * modes;
}

__global__ void __launch_bounds__(256) power_bin_kernel(const float2* __restrict__ spec, int m, double ell_scale,
                                                        double p_norm, int nbins,
                                                        const __grid_constant__ PowerEdges edges,
                                                        double* __restrict__ sums) {
  extern __shared__ double sh[];  // [3][nbins]
  __shared__ int edge[PowerEdges::kMaxBins + 1];
  for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x) sh[i] = 0.0;
  for (int i = threadIdx.x; i <= nbins; i += blockDim.x) edge[i] = edges.first[i];
  __syncthreads();
  const int mzc = m / 2 + 1, segments = (mzc + kBinColumns - 1) / kBinColumns, lane = threadIdx.x & 31;
  const int task = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nx = task / segments, z0 = (task - nx * segments) * kBinColumns + lane;
  if (nx <= m / 2) {
    const bool two = nx > 0 && nx < m / 2;
    const float2* __restrict__ row = spec + static_cast<int64_t>(nx) * mzc;
    const float2* __restrict__ mirror = spec + static_cast<int64_t>(m - nx) * mzc;
    const float2 none = make_float2(0.f, 0.f);
    float2 u[kBinColumns / 32], v[kBinColumns / 32];
#pragma unroll
    for (int i = 0; i < kBinColumns / 32; ++i) {
      const int iz = z0 + 32 * i;
      u[i] = iz < mzc ? __ldg(row + iz) : none;
      v[i] = two && iz < mzc ? __ldg(mirror + iz) : none;
    }
    // the bin below the first mode's: the last whose first |n|^2 is not above it, -1 below all
    int bin = -1;
    {
      const int n2 = nx * nx + z0 * z0;
      for (int lo = 0, hi = nbins; lo <= hi;) {
        const int mid = (lo + hi) >> 1;
        if (edge[mid] <= n2) {
          bin = mid;
          lo = mid + 1;
        } else {
          hi = mid - 1;
        }
      }
    }
    // squares in floats where no square or its rounding error can leave float's range, else in FP64
    bool small = true;
#pragma unroll
    for (int i = 0; i < kBinColumns / 32; ++i) small = small && moderate(u[i]) && moderate(v[i]);
    const bool plain = __all_sync(0xffffffffu, small);
    double power = 0.0;
    Sum3 squares{0.f, 0.f, 0.f}, roots{0.f, 0.f, 0.f};
    int count = 0;
    // what the lanes with `out` hold of their bins, summed over the lanes of the same bin; by the whole warp
    auto drain = [&](bool out) {
      const double ell = value(roots) * ell_scale, all = (power + value(squares)) * p_norm;
      unsigned left = __ballot_sync(0xffffffffu, out && count > 0 && bin >= 0 && bin < nbins);
      while (left) {
        const int leader = __ffs(left) - 1;
        const int leading = __shfl_sync(0xffffffffu, bin, leader);  // by every lane: not behind a short circuit
        const bool mine = ((left >> lane) & 1u) && bin == leading;
        double p = mine ? all : 0.0, e = mine ? ell : 0.0;
        int c = mine ? count : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          p += __shfl_xor_sync(0xffffffffu, p, o);
          e += __shfl_xor_sync(0xffffffffu, e, o);
          c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (lane == leader) {
          atomicAdd(sh + bin, p);
          atomicAdd(sh + nbins + bin, e);
          atomicAdd(sh + 2 * nbins + bin, static_cast<double>(c));
        }
        left &= ~__ballot_sync(0xffffffffu, mine);
      }
      if (out) {
        power = 0.0;
        squares = roots = Sum3{0.f, 0.f, 0.f};
        count = 0;
      }
    };
#pragma unroll
    for (int i = 0; i < kBinColumns / 32; ++i) {
      const int iz = z0 + 32 * i;
      const int n2 = nx * nx + iz * iz;
      const bool mode = iz < mzc && n2 > 0;
      const bool next = mode && bin < nbins && n2 >= edge[bin + 1];
      if (__any_sync(0xffffffffu, next)) {
        drain(next);
        if (next) {
          do ++bin;
          while (bin < nbins && n2 >= edge[bin + 1]);
        }
        __syncwarp();
      }
      if (mode) {
        const int each = iz == 0 || iz == m / 2 ? 1 : 2, modes = two ? 2 * each : each;
        const float scale = static_cast<float>(each);
        if (plain) {
          add_square(squares, u[i].x, scale);
          add_square(squares, u[i].y, scale);
          if (two) {
            add_square(squares, v[i].x, scale);
            add_square(squares, v[i].y, scale);
          }
        } else {
          double pw = static_cast<double>(u[i].x) * u[i].x + static_cast<double>(u[i].y) * u[i].y;
          if (two) pw += static_cast<double>(v[i].x) * v[i].x + static_cast<double>(v[i].y) * v[i].y;
          power += each == 2 ? 2.0 * pw : pw;
        }
        count += modes;
        add_root(roots, n2, modes);
      }
      __syncwarp();
    }
    drain(true);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x)
    if (sh[i] != 0.0) atomicAdd(sums + i, sh[i]);
}

PowerEdges power_edges(int64_t m, double dtheta, int nbins, double ell_min, double ell_max) {
  const double theta_field = m * dtheta, ln_lmin = std::log(ell_min), inv_ln_ratio = 1.0 / std::log(ell_max / ell_min);
  const int64_t none = m * m / 2 + 1;  // above every |n|^2
  auto rule = [&](int64_t n2) {
    return nbins * (std::log(2.0 * M_PI * std::sqrt(static_cast<double>(n2)) / theta_field) - ln_lmin) * inv_ln_ratio + 1e-9;
  };
  PowerEdges e{};
  for (int b = 0; b <= nbins; ++b) {
    // next to where the rule's inverse puts it, else (its rounding, or an overflow) by bisection
    const double ell = std::exp(ln_lmin + (b - 1e-9) / (nbins * inv_ln_ratio)), n = ell * theta_field / (2.0 * M_PI);
    int64_t lo = 0, hi = none;  // the rule fails at lo and holds at hi, or hi is past the end
    if (std::isfinite(inv_ln_ratio)) {
      if (n * n < static_cast<double>(none)) {
        const int64_t c = static_cast<int64_t>(n * n);
        if (c > 1 && !(rule(c - 1) >= b)) lo = c - 1;
        if (c + 2 < none && rule(c + 2) >= b) hi = c + 2;
      }
      while (hi - lo > 1) {
        const int64_t c = lo + (hi - lo) / 2;
        if (rule(c) >= b) hi = c;
        else lo = c;
      }
    }
    e.first[b] = static_cast<int>(hi);
  }
  return e;
}

hrt_status launch_power_bin(const void* spec, int64_t m, double dtheta, int nbins, double ell_min, double ell_max,
                            double* sums, cudaStream_t s) {
  HRT_CUDA(cudaMemsetAsync(sums, 0, 3 * nbins * sizeof(double), s));
  const double theta_field = m * dtheta;
  // |FFT|^2 dtheta^4 / Theta^2
  const double p_norm = dtheta * dtheta * dtheta * dtheta / (theta_field * theta_field);
  const int64_t warps = (m / 2 + 1) * ((m / 2 + 1 + kBinColumns - 1) / kBinColumns);
  power_bin_kernel<<<blocks_for(warps, 8), 256, 3 * nbins * sizeof(double), s>>>(
      static_cast<const float2*>(spec), static_cast<int>(m), 2.0 * M_PI / theta_field, p_norm, nbins,
      power_edges(m, dtheta, nbins, ell_min, ell_max), sums);
  HRT_LAUNCHED("power_bin_kernel");
  return HRT_OK;
}

}  // namespace hrt
