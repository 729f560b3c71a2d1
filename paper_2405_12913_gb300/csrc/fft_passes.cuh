// The split Poisson solve: FFT passes along z, y and x, the k-space step inside the x-pass, and back.
//
// What bounds it.  A 3D transform has to cross memory once per axis, because a line along the next axis needs every
// block's output of the last one.  The passes here read and write each spectrum once per axis and nothing else: at
// 1024^3 8.7 GB forward along z, 8.7 GB along y, 13.1 GB along x (two spectra out of one: see below), 21.8 GB inverse
// along y (three fields out of two) and 26 GB along z.  cuFFT's batched 2D plans cross memory twice per transform
// on top of that, and the gradient's three components took three inverse transforms along x.
//
// Two spectra out of the x-pass.  The gradient spectra of one filter set are i k_j c X.  Along x only the x component
// has its own factor; d_y and d_z are constant on an x line.  So the x-pass writes IFFT_x(i c d_x X) and
// V = IFFT_x(i c X), the inverse y-pass makes IFFT_y(d_y V) and d_z IFFT_y(V) out of V, and the inverse z-pass
// finishes three fields.
//
// Layouts.  Rows [x][y][kz] between the z- and y-passes (row: kz in pairs, (re, re, im, im) of kz and kz + 1, padded to
// a multiple of 8 columns), and tiles [ky / 16][kz / 8][x][ky mod 16][kz mod 8] between the y- and x-passes: a chunk of
// 16 ky x 8 kz is 1 KB.  A y tile (one x, 8 kz, every y) reads rows of 64 B that its neighbours complete to full lines
// and writes 1 KB chunks; an x tile (one ky, 8 kz, every x) lies in one region of n KB.  No pass touches rows
// megabytes apart, which had held the former x-pass at a third of the copy rate (its rows of 64 B lay one per 2 MB
// page).  Copies of this shape by TMA alone run at 6.8-7.2 TB/s on a GB300.
//
// Sides are 32 R1 with R1 in {2, 3, 4, 6, 8, 12, 16, 24, 32}.  FFT of n = 32 R1 points in a warp, four-step with x = l + 32 m and k = k1 + R1 k2: lane l holds x = l + 32 m of P lines, does R1-point
// DFTs over m in registers, multiplies by W_n^(l k1), and an exchange through shared memory gives lane (p, k1) the 32
// values over l, whose 32-point DFT leaves X[k1 + R1 k2].  Every lane carries two lines side by side in packed
// FP32 pairs (add/mul/fma.f32x2: one instruction for both), which are two neighbouring kz columns in the y- and
// x-passes and two pairs of real rows in the z-passes; a complex pair is 16 bytes, so each shared-memory access is a
// 16-byte one without bank conflicts.  A warp exchanges through the shared memory that holds its own columns, so the
// block synchronises only around the tile's copies, and 64 KB tiles leave room for three blocks of four warps per SM
// (168 registers a thread): one block computes while the copies of the others are in flight.
//
// The inverse transform is the forward one with the real and imaginary parts swapped on both sides.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "common.h"
#include "fft_passes.h"
#include "packed.cuh"
#include "tma.h"

namespace hrt {

namespace {

using namespace tma;
// Two complex numbers side by side, 16 bytes in memory: (re, re, im, im).
struct C2 {
  u64 re, im;
};
__device__ __forceinline__ C2 operator+(C2 a, C2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 operator-(C2 a, C2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ C2 swapped(C2 a) { return {a.im, a.re}; }
// v (c - i s)
__device__ __forceinline__ C2 turn(C2 v, u64 c, u64 s, u64 neg_s) {
  return {fma2(v.re, c, mul2(v.im, s)), fma2(v.im, c, mul2(v.re, neg_s))};
}

__device__ __forceinline__ C2 lds(uint32_t a) {
  C2 v;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v.re), "=l"(v.im) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts(uint32_t a, C2 v) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(a), "l"(v.re), "l"(v.im) : "memory");
}

// Streamed inputs bypass L1, which is left to the twiddles.
__device__ __forceinline__ float stream_load(const float* p) {
  float v;
  asm volatile("ld.global.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 stream_load4(const float* p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}

// ---- DFTs in registers --------------------------------------------------------------------------------------
// (cos, sin) of 2 pi t / 32, t in [0, 32): FP64 values rounded to float.
__device__ __forceinline__ constexpr float cos32(int t) {
  constexpr float c[9] = {1.f,
                          9.807852804e-01f,
                          9.238795325e-01f,
                          8.314696123e-01f,
                          7.071067812e-01f,
                          5.555702330e-01f,
                          3.826834324e-01f,
                          1.950903220e-01f,
                          0.f};
  const int u = t & 31, q = u > 16 ? 32 - u : u;
  return q > 8 ? -c[16 - q] : c[q];
}
// (cos, sin) of 2 pi t / 24
__device__ __forceinline__ constexpr float cos24(int t) {
  constexpr float c[7] = {1.f, 9.659258263e-01f, 8.660254038e-01f, 7.071067812e-01f, 0.5f, 2.588190451e-01f, 0.f};
  const int u = t % 24, q = u > 12 ? 24 - u : u;
  return q > 6 ? -c[12 - q] : c[q];
}
// of 2 pi t / R, R a divisor of 32 or 24
template <int R>
__device__ __forceinline__ constexpr float cos_of(int t) {
  return 32 % R == 0 ? cos32(t * (32 / R)) : cos24(t * (24 / R));
}
template <int R>
__device__ __forceinline__ constexpr float sin_of(int t) {
  return 32 % R == 0 ? cos32(t * (32 / R) + 24) : cos24(t * (24 / R) + 18);
}

__device__ __forceinline__ void dft2(C2& a, C2& b) {
  const C2 t = a - b;
  a = a + b;
  b = t;
}

__device__ __forceinline__ void dft3(C2& a, C2& b, C2& c) {
  const u64 h = both(-0.5f), s = both(8.660254038e-01f), ns = both(-8.660254038e-01f);
  const C2 t = b + c, d = b - c, m = {fma2(t.re, h, a.re), fma2(t.im, h, a.im)};
  a = a + t;
  b = {fma2(d.im, s, m.re), fma2(d.re, ns, m.im)};
  c = {fma2(d.im, ns, m.re), fma2(d.re, s, m.im)};
}

__device__ __forceinline__ void dft4(C2& a, C2& b, C2& c, C2& d) {
  const C2 s0 = a + c, d0 = a - c, s1 = b + d, d1 = b - d;
  a = s0 + s1;
  c = s0 - s1;
  b = {add2(d0.re, d1.im), sub2(d0.im, d1.re)};
  d = {sub2(d0.re, d1.im), add2(d0.im, d1.re)};
}

__device__ __forceinline__ void dft8(C2& v0, C2& v1, C2& v2, C2& v3, C2& v4, C2& v5, C2& v6, C2& v7) {
  const C2 a0 = v0 + v4, a1 = v0 - v4, a2 = v2 + v6, a3 = v2 - v6;
  const C2 b0 = v1 + v5, b1 = v1 - v5, b2 = v3 + v7, b3 = v3 - v7;
  const C2 e0 = a0 + a2, e1 = a0 - a2, f0 = b0 + b2, f1 = b0 - b2;
  v0 = e0 + f0;
  v4 = e0 - f0;
  v2 = {add2(e1.re, f1.im), sub2(e1.im, f1.re)};
  v6 = {sub2(e1.re, f1.im), add2(e1.im, f1.re)};
  const C2 p = {add2(a1.re, a3.im), sub2(a1.im, a3.re)}, q = {add2(b1.re, b3.im), sub2(b1.im, b3.re)};
  const C2 r = {sub2(a1.re, a3.im), add2(a1.im, a3.re)}, s = {sub2(b1.re, b3.im), add2(b1.im, b3.re)};
  const u64 h = both(7.071067812e-01f), nh = both(-7.071067812e-01f);
  // v1, v5 = p +- (1 - i) q / sqrt 2;  v3, v7 = r -+ (1 + i) s / sqrt 2
  const u64 q0 = add2(q.re, q.im), q1 = sub2(q.im, q.re), s0 = sub2(s.im, s.re), s1 = add2(s.re, s.im);
  v1 = {fma2(h, q0, p.re), fma2(h, q1, p.im)};
  v5 = {fma2(nh, q0, p.re), fma2(nh, q1, p.im)};
  v3 = {fma2(h, s0, r.re), fma2(nh, s1, r.im)};
  v7 = {fma2(nh, s0, r.re), fma2(h, s1, r.im)};
}

// R = A B points v[OFF ..): R-point DFT in place, X[k] left in register slot OFF + slot<R>(k).
template <int R>
struct Split {
  static constexpr int B = R % 8 == 0 && R != 16 ? 8 : R % 4 == 0 ? 4 : R % 3 == 0 ? 3 : 2;
  static constexpr int A = R / B;
};

template <int R>
__host__ __device__ constexpr int slot(int k) {
  return Split<R>::B * (k % Split<R>::A) + k / Split<R>::A;
}

template <int R, int OFF>
__device__ __forceinline__ void dft(C2 (&v)[32]) {
  constexpr int A = Split<R>::A, B = Split<R>::B;
  static_assert(A <= 4 && A * B == R);
  if constexpr (A > 1) {
#pragma unroll
    for (int b = 0; b < B; ++b) {
      C2* w = &v[OFF + b];
      if constexpr (A == 2) dft2(w[0], w[B]);
      else if constexpr (A == 3) dft3(w[0], w[B], w[2 * B]);
      else dft4(w[0], w[B], w[2 * B], w[3 * B]);
    }
#pragma unroll
    for (int c = 1; c < A; ++c)
#pragma unroll
      for (int b = 1; b < B; ++b) {
        const int t = b * c;
        C2& x = v[OFF + B * c + b];
        if (4 * t == R) x = {x.im, sub2(both(0.f), x.re)};
        else x = turn(x, both(cos_of<R>(t)), both(sin_of<R>(t)), both(-sin_of<R>(t)));
      }
  }
#pragma unroll
  for (int c = 0; c < A; ++c) {
    C2* w = &v[OFF + B * c];
    if constexpr (B == 8) dft8(w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
    else if constexpr (B == 4) dft4(w[0], w[1], w[2], w[3]);
    else if constexpr (B == 3) dft3(w[0], w[1], w[2]);
    else dft2(w[0], w[1]);
  }
}

template <int R, int P>
struct Dfts {
  __device__ __forceinline__ static void run(C2 (&v)[32]) {
    dft<R, (P - 1) * R>(v);
    Dfts<R, P - 1>::run(v);
  }
};
template <int R>
struct Dfts<R, 0> {
  __device__ __forceinline__ static void run(C2 (&)[32]) {}
};

// ---- lines of a warp ----------------------------------------------------------------------------------------
// P line pairs per warp and W warps per tile: 4 pairs (8 kz) per tile row.
template <int R1>
struct Cfg {
  static constexpr int N = 32 * R1;
  static constexpr int P = R1 > 16 ? 1 : R1 > 8 ? 2 : 4;
  static constexpr int W = 4 / P;
  static constexpr int Threads = 32 * W;
  static constexpr int Blocks = 12 / W;  // resident per SM: 12 warps of up to 168 registers a thread
  static constexpr int TileBytes = N * 64;
  static constexpr int Rows = N <= 256 ? N : N % 256 == 0 ? 256 : 128;  // rows per TMA box
  static constexpr int Boxes = N / Rows;
  // lane's place among the P R1 that hold a k1 each; the others do the work of one of them again (the same values to
  // the same places)
  __device__ __forceinline__ static int second(int lane) { return lane % (P * R1); }
};

// Address of pair p's element r.  TileAddr: rows of 64 bytes (4 pairs of 16 bytes) under the 64-byte TMA swizzle, a
// warp's pairs starting at column c0; 8 consecutive r cover all 32 banks.  RowAddr: a warp's lines one after another.
struct TileAddr {
  uint32_t base;
  int c0;
  __device__ __forceinline__ uint32_t operator()(int p, int r) const {
    return base + r * 64 + (((c0 + p) ^ ((r >> 1) & 3)) << 4);
  }
};
template <int N>
struct RowAddr {
  uint32_t base;
  __device__ __forceinline__ uint32_t operator()(int p, int r) const { return base + (p * N + r) * 16; }
  // natural order with neighbouring even elements on different banks
  __device__ __forceinline__ uint32_t natural(int p, int k) const { return (*this)(p, k ^ ((k >> 3) & 1)); }
};

// Exchange slot of (k1, l): rows of 32 whose low bits are XORed with k1, so that a warp's accesses along either index
// fall on different banks.
__device__ __forceinline__ int exchange(int k1, int l) { return k1 * 32 + (l ^ (k1 & 7)); }

__device__ __forceinline__ C2 twiddled(C2 v, float2 t) { return turn(v, both(t.x), both(t.y), both(-t.y)); }

// Forward: v[p R1 + m] = x[lane + 32 m] of pair p -> v[slot<32>(k2)] = X[k1 + R1 k2] of pair lane / R1.
template <int R1, class Addr>
__device__ __forceinline__ void forward_lines(C2 (&v)[32], const Addr& at, const float2* __restrict__ tw, int lane) {
  constexpr int P = Cfg<R1>::P;
  Dfts<R1, P>::run(v);
#pragma unroll
  for (int k1 = 1; k1 < R1; ++k1) {
    const float2 t = __ldg(tw + k1 * 32 + lane);
#pragma unroll
    for (int p = 0; p < P; ++p) v[p * R1 + slot<R1>(k1)] = twiddled(v[p * R1 + slot<R1>(k1)], t);
  }
  __syncwarp();
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) sts(at(p, exchange(k1, lane)), v[p * R1 + slot<R1>(k1)]);
  __syncwarp();
  const int lb = Cfg<R1>::second(lane), pb = lb / R1, k1 = lb % R1;
#pragma unroll
  for (int l = 0; l < 32; ++l) v[l] = lds(at(pb, exchange(k1, l)));
  __syncwarp();
  dft<32, 0>(v);
}

// Inverse of forward_lines (unnormalised): v[k2] = X[k1 + R1 k2] of pair lane / R1, real and imaginary parts swapped
// -> v[p R1 + slot<R1>(n2)] = x[lane + 32 n2] of pair p, still swapped.  The first half works in registers only.
template <int R1>
__device__ __forceinline__ void inverse_first(C2 (&v)[32], const float2* __restrict__ tw, int lane) {
  dft<32, 0>(v);
  const float2* __restrict__ ti = tw + (R1 == 32 ? 0 : R1 * 32);
#pragma unroll
  for (int n1 = 1; n1 < 32; ++n1) v[slot<32>(n1)] = twiddled(v[slot<32>(n1)], __ldg(ti + n1 * 32 + lane));
}
template <int R1, class Addr>
__device__ __forceinline__ void inverse_second(C2 (&v)[32], const Addr& at, int lane) {
  constexpr int P = Cfg<R1>::P;
  const int lb = Cfg<R1>::second(lane), pb = lb / R1, k1 = lb % R1;
  __syncwarp();
#pragma unroll
  for (int n1 = 0; n1 < 32; ++n1) sts(at(pb, exchange(k1, n1)), v[slot<32>(n1)]);
  __syncwarp();
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int j = 0; j < R1; ++j) v[p * R1 + j] = lds(at(p, exchange(j, lane)));
  __syncwarp();
  Dfts<R1, P>::run(v);
}

// ---- z-passes -----------------------------------------------------------------------------------------------
struct ZFields {
  const float* in[kFftMaxFields];
  float* out[kFftMaxFields];
};

struct ZForward {
  float* in[2];  // zeroed once read, on request
  float* out[2];
};

// A warp takes P groups of four consecutive rows; a group's lines are row 0 + i row 1 and row 2 + i row 3.
// Forward: bound by memory (8.7 GB, with the zeroing 13 GB at 1024^3).
template <int R1>
__global__ void __launch_bounds__(128, 3)
    fft_z_kernel(const __grid_constant__ ZForward f, const float2* __restrict__ tw, int groups, int row_out, bool clear) {
  constexpr int N = 32 * R1, P = Cfg<R1>::P;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t g0 = (static_cast<int64_t>(blockIdx.x) * 4 + warp) * P;
  if (g0 >= groups) return;
  const RowAddr<N> at{smem_u32(smem) + warp * (P * N * 16)};
  float* __restrict__ src = f.in[blockIdx.y] + g0 * 4 * N;
  float* __restrict__ out = f.out[blockIdx.y];
  C2 v[32];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const float* q = src + p * 4 * N + lane + 32 * m;
      v[p * R1 + m] = {pack(stream_load(q), stream_load(q + 2 * N)), pack(stream_load(q + N), stream_load(q + 3 * N))};
    }
  forward_lines<R1>(v, at, tw, lane);
  const int lb = Cfg<R1>::second(lane), pb = lb / R1, k1 = lb % R1;
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) sts(at.natural(pb, k1 + R1 * k2), v[slot<32>(k2)]);
  __syncwarp();
  if (clear) {
    float4* z = reinterpret_cast<float4*>(src);
#pragma unroll 4
    for (int i = lane; i < P * N; i += 32) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // two lines of real rows a + i b: A[k] = (X[k] + conj X[n-k]) / 2, B[k] = (X[k] - conj X[n-k]) / 2i
  const u64 hp = both(0.5f), hn = both(-0.5f);
#pragma unroll 1
  for (int p = 0; p < P; ++p) {
    float* dst = out + (g0 + p) * 4 * static_cast<int64_t>(row_out);
    constexpr int J = (N / 4 + 31) / 32;
#pragma unroll(J < 4 ? J : J % 4 == 0 ? 4 : 3)
    for (int t = 0; t < J; ++t) {
      const int j = lane + 32 * t;
      if (N % 128 != 0 && j >= N / 4) break;
      C2 a[2], b[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int k = 2 * j + i;
        const C2 x = lds(at.natural(p, k)), y = lds(at.natural(p, k == 0 ? 0 : N - k));
        const u64 xr = mul2(x.re, hp), xi = mul2(x.im, hp);
        a[i] = {fma2(y.re, hp, xr), fma2(y.im, hn, xi)};
        b[i] = {fma2(y.im, hp, xi), fma2(x.re, hn, mul2(y.re, hp))};
      }
      const float2 ar0 = unpack(a[0].re), ar1 = unpack(a[1].re), ai0 = unpack(a[0].im), ai1 = unpack(a[1].im);
      const float2 br0 = unpack(b[0].re), br1 = unpack(b[1].re), bi0 = unpack(b[0].im), bi1 = unpack(b[1].im);
      float* q = dst + 4 * j;
      *reinterpret_cast<float4*>(q) = make_float4(ar0.x, ar1.x, ai0.x, ai1.x);
      *reinterpret_cast<float4*>(q + row_out) = make_float4(br0.x, br1.x, bi0.x, bi1.x);
      *reinterpret_cast<float4*>(q + 2 * row_out) = make_float4(ar0.y, ar1.y, ai0.y, ai1.y);
      *reinterpret_cast<float4*>(q + 3 * row_out) = make_float4(br0.y, br1.y, bi0.y, bi1.y);
    }
    if (lane < 4) {  // k = n/2 of the four rows
      const C2 x = lds(at.natural(p, N / 2));
      const float2 v2 = unpack(lane & 1 ? x.im : x.re);
      *reinterpret_cast<float4*>(dst + lane * row_out + N) = make_float4(lane & 2 ? v2.y : v2.x, 0.f, 0.f, 0.f);
    }
  }
}

// Inverse: the imaginary parts of k = 0 and n/2 do not count, as in any complex-to-real transform.
template <int R1>
__global__ void __launch_bounds__(128, 3)
    fft_iz_kernel(const __grid_constant__ ZFields f, const float2* __restrict__ tw, int groups, int row_in) {
  constexpr int N = 32 * R1, P = Cfg<R1>::P;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t g0 = (static_cast<int64_t>(blockIdx.x) * 4 + warp) * P;
  if (g0 >= groups) return;
  const RowAddr<N> at{smem_u32(smem) + warp * (P * N * 16)};
  const float* __restrict__ in = f.in[blockIdx.y] + g0 * 4 * static_cast<int64_t>(row_in);
  // every load of the warp's rows in flight at once: 4 rows x (n / 128) x 16 bytes per lane and group
  constexpr int J = (N / 4 + 31) / 32;
  float4 r[P * J][4];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int i = 0; i < J; ++i)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (N % 128 == 0 || lane + 32 * i < N / 4)
          r[p * J + i][k] = stream_load4(in + (4 * p + k) * row_in + 4 * (lane + 32 * i));
  float nyq[P];
#pragma unroll
  for (int p = 0; p < P; ++p) nyq[p] = lane < 4 ? stream_load(in + (4 * p + lane) * row_in + N) : 0.f;
#pragma unroll
  for (int p = 0; p < P; ++p) {
#pragma unroll
    for (int i = 0; i < J; ++i) {
      if (N % 128 != 0 && lane + 32 * i >= N / 4) continue;
      // (row 0, row 2) and (row 1, row 3) at k = 2j and 2j + 1: C = A + i B, C[n - k] = conj A + i conj B
      const float4 r0 = r[p * J + i][0], r1 = r[p * J + i][1], r2 = r[p * J + i][2], r3 = r[p * J + i][3];
      const u64 ar[2] = {pack(r0.x, r2.x), pack(r0.y, r2.y)}, ai[2] = {pack(r0.z, r2.z), pack(r0.w, r2.w)};
      const u64 br[2] = {pack(r1.x, r3.x), pack(r1.y, r3.y)}, bi[2] = {pack(r1.z, r3.z), pack(r1.w, r3.w)};
      const int k = 2 * (lane + 32 * i);
      if (k == 0) {
        sts(at.natural(p, 0), {ar[0], br[0]});
      } else {
        sts(at.natural(p, k), {sub2(ar[0], bi[0]), add2(ai[0], br[0])});
        sts(at.natural(p, N - k), {add2(ar[0], bi[0]), sub2(br[0], ai[0])});
      }
      sts(at.natural(p, k + 1), {sub2(ar[1], bi[1]), add2(ai[1], br[1])});
      sts(at.natural(p, N - k - 1), {add2(ar[1], bi[1]), sub2(br[1], ai[1])});
    }
    // k = n/2 of the four rows, one per lane
    const float n1 = __shfl_sync(0xffffffffu, nyq[p], 1), n2 = __shfl_sync(0xffffffffu, nyq[p], 2),
                n3 = __shfl_sync(0xffffffffu, nyq[p], 3);
    if (lane == 0) sts(at.natural(p, N / 2), {pack(nyq[p], n2), pack(n1, n3)});
  }
  __syncwarp();
  const int lb = Cfg<R1>::second(lane), pb = lb / R1, k1 = lb % R1;
  C2 v[32];
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) v[k2] = swapped(lds(at.natural(pb, k1 + R1 * k2)));
  inverse_first<R1>(v, tw, lane);
  inverse_second<R1>(v, at, lane);
  float* __restrict__ dst = f.out[blockIdx.y] + g0 * 4 * N;
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      float* q = dst + p * 4 * N + lane + 32 * m;
      const C2 x = v[p * R1 + slot<R1>(m)];
      const float2 re = unpack(x.im), im = unpack(x.re);
      q[0] = re.x;
      q[N] = im.x;
      q[2 * N] = re.y;
      q[3 * N] = im.y;
    }
}

// ---- tile copies --------------------------------------------------------------------------------------------
__device__ __forceinline__ void load_5d(uint32_t dst, const CUtensorMap* map, int c1, int c2, int c3, int c4,
                                        uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, "
      "%6}], [%7];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void store_5d(const CUtensorMap* map, uint32_t src, int c1, int c2, int c3, int c4) {
  asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];\n" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
               : "memory");
}
__device__ __forceinline__ void store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];\n" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(c0), "r"(c1)
               : "memory");
}

// A tile as each pass sees it: rows of a plane (Plane), the ky rows of an x (Column) or the x rows of a ky (Line).
template <int R1>
struct Tile {
  using C = Cfg<R1>;
  __device__ __forceinline__ static void load_plane(uint32_t dst, const CUtensorMap* m, int x, int kb, uint32_t bar) {
#pragma unroll
    for (int i = 0; i < C::Boxes; ++i) load_2d(dst + i * C::Rows * 64, m, 16 * kb, x * C::N + i * C::Rows, bar);
  }
  __device__ __forceinline__ static void store_plane(const CUtensorMap* m, uint32_t src, int x, int kb) {
#pragma unroll
    for (int i = 0; i < C::Boxes; ++i) store_2d(m, src + i * C::Rows * 64, 16 * kb, x * C::N + i * C::Rows);
  }
  __device__ __forceinline__ static void load_column(uint32_t dst, const CUtensorMap* m, int x, int kb, uint32_t bar) {
#pragma unroll
    for (int i = 0; i < C::Boxes; ++i) load_5d(dst + i * C::Rows * 64, m, 0, x, kb, i * (C::Rows / 16), bar);
  }
  __device__ __forceinline__ static void store_column(const CUtensorMap* m, uint32_t src, int x, int kb) {
#pragma unroll
    for (int i = 0; i < C::Boxes; ++i) store_5d(m, src + i * C::Rows * 64, 0, x, kb, i * (C::Rows / 16));
  }
  __device__ __forceinline__ static void load_line(uint32_t dst, const CUtensorMap* m, int ky, int kb, uint32_t bar) {
#pragma unroll
    for (int i = 0; i < C::Boxes; ++i) load_5d(dst + i * C::Rows * 64, m, ky & 15, i * C::Rows, kb, ky >> 4, bar);
  }
  __device__ __forceinline__ static void store_line(const CUtensorMap* m, uint32_t src, int ky, int kb) {
#pragma unroll
    for (int i = 0; i < C::Boxes; ++i) store_5d(m, src + i * C::Rows * 64, ky & 15, i * C::Rows, kb, ky >> 4);
  }
};

// A warp's tile within its block of G tiles: the tile's number, buffer (1024-byte aligned) and barrier, the warp among the
// tile's and the thread that issues its copies.
template <int R1, int G = 1>
struct Place {
  using C = Cfg<R1>;
  const unsigned char* raw;
  uint64_t* bars;
  __device__ __forceinline__ static int group() { return G == 1 ? 0 : static_cast<int>(threadIdx.x) / C::Threads; }
  __device__ __forceinline__ unsigned tile() const { return blockIdx.x * G + group(); }
  __device__ __forceinline__ uint32_t base() const { return (smem_u32(raw) + 1023u) & ~1023u; }
  __device__ __forceinline__ uint32_t buf() const { return base() + group() * C::TileBytes; }
  __device__ __forceinline__ uint32_t bar() const { return smem_u32(bars + group()); }
  __device__ __forceinline__ int warp() const { return static_cast<int>(threadIdx.x >> 5) - group() * C::W; }
  __device__ __forceinline__ bool leader() const { return (G == 1 ? threadIdx.x : threadIdx.x % C::Threads) == 0; }
};

// One tile's copy into its buffer; load(dst, bar) issues the copies.  False for the whole block after a timed-out wait, with
// the copies given another bounded wait to land before the block ends.
template <int R1, int G, class Load>
__device__ __forceinline__ bool fetch_tile(const Place<R1, G>& at, int* __restrict__ err, Load load) {
  const uint32_t b = at.bar(), buf = at.buf();
  if (at.leader()) {
    mbar_init(b, 1);
    fence_mbar_init();
    mbar_expect_tx(b, Cfg<R1>::TileBytes);
    load(buf, b);
  }
  __syncthreads();
  const bool got = mbar_wait(b, 0u);
  if (__syncthreads_and(got)) return true;
  if (at.leader()) {
    atomicOr(err, kFftTimeout);
    mbar_wait(b, 0u);
  }
  return false;
}

// The next tile into the buffer once every warp is done with the last one; phase: its number, from 1.
template <int R1, int G, class Load>
__device__ __forceinline__ bool fetch_next(const Place<R1, G>& at, uint32_t phase, int* __restrict__ err, Load load) {
  const uint32_t b = at.bar(), buf = at.buf();
  fence_async_shared();
  __syncthreads();
  if (at.leader()) {
    mbar_expect_tx(b, Cfg<R1>::TileBytes);
    load(buf, b);
  }
  const bool got = mbar_wait(b, phase & 1u);
  if (__syncthreads_and(got)) return true;
  if (at.leader()) {
    atomicOr(err, kFftTimeout);
    mbar_wait(b, phase & 1u);
  }
  return false;
}

// Signed frequency times kf, 0 at the Nyquist frequency.
__device__ __forceinline__ float derivative(int k, int n, float kf) {
  const int s = k < (n >> 1) ? k : k - n;
  return s == -(n >> 1) ? 0.f : kf * s;
}

// ---- y-passes -----------------------------------------------------------------------------------------------
struct YForward {
  CUtensorMap in[2], out[2];
};

// Forward: rows of plane x -> column tile.  One block per (x, 8 kz).
template <int R1>
__global__ void __launch_bounds__(Cfg<R1>::Threads, Cfg<R1>::Blocks)
    fft_y_kernel(const __grid_constant__ YForward f, const float2* __restrict__ tw, int blocks_kz, int* __restrict__ err) {
  using C = Cfg<R1>;
  using T = Tile<R1>;
  extern __shared__ unsigned char raw[];
  __shared__ uint64_t bars[1];
  const Place<R1> here{raw, bars};
  const uint32_t buf = here.buf();
  const int x = here.tile() / blocks_kz, kb = here.tile() - x * blocks_kz;
  if (!fetch_tile(here, err, [&](uint32_t d, uint32_t b) { T::load_plane(d, &f.in[blockIdx.y], x, kb, b); })) return;
  const int lane = threadIdx.x & 31, warp = here.warp();
  const TileAddr at{buf, warp * C::P};
  C2 v[32];
#pragma unroll
  for (int p = 0; p < C::P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) v[p * R1 + m] = lds(at(p, lane + 32 * m));
  forward_lines<R1>(v, at, tw, lane);
  const int lb = Cfg<R1>::second(lane), pb = lb / R1, k1 = lb % R1;
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) sts(at(pb, k1 + R1 * k2), v[slot<32>(k2)]);
  fence_async_shared();
  __syncthreads();
  if (here.leader()) {
    T::store_column(&f.out[blockIdx.y], buf, x, kb);
    bulk_commit();
    bulk_wait_read_all();
  }
}

struct YJobs {
  CUtensorMap in[kFftMaxFields], out[kFftMaxFields];
  int jobs;
};

// Inverse: column tile -> rows of plane x.  Per filter set three jobs in neighbouring blocks: the x component as it is,
// d_y V before the transform (job 1), d_z V after it (job 2); the second reading of V hits L2.
template <int R1>
__global__ void __launch_bounds__(Cfg<R1>::Threads, Cfg<R1>::Blocks)
    fft_iy_kernel(const __grid_constant__ YJobs jobs, const float2* __restrict__ tw, int blocks_kz, float kf,
                  int* __restrict__ err) {
  using C = Cfg<R1>;
  using T = Tile<R1>;
  extern __shared__ unsigned char raw[];
  __shared__ uint64_t bars[1];
  const Place<R1> here{raw, bars};
  const uint32_t buf = here.buf();
  const unsigned tile = here.tile() / static_cast<unsigned>(jobs.jobs);
  const int job = here.tile() - tile * jobs.jobs;
  const int x = tile / blocks_kz, kb = tile - x * blocks_kz;
  if (!fetch_tile(here, err, [&](uint32_t d, uint32_t b) { T::load_column(d, &jobs.in[job], x, kb, b); })) return;
  const int lane = threadIdx.x & 31, warp = here.warp();
  const TileAddr at{buf, warp * C::P};
  const int kind = job % 3;
  C2 v[32];
#pragma unroll
  for (int p = 0; p < C::P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) v[p * R1 + m] = swapped(lds(at(p, lane + 32 * m)));
  if (kind == 1) {
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const u64 d = both(derivative(lane + 32 * m, C::N, kf));
#pragma unroll
      for (int p = 0; p < C::P; ++p) v[p * R1 + m] = {mul2(v[p * R1 + m].re, d), mul2(v[p * R1 + m].im, d)};
    }
  }
  forward_lines<R1>(v, at, tw, lane);
  const int lb = Cfg<R1>::second(lane), pb = lb / R1, k1 = lb % R1;
  if (kind == 2) {
    const int kz = kb * 8 + 2 * (warp * C::P + pb);
    const u64 d = pack(kz == C::N / 2 ? 0.f : kf * kz, kf * (kz + 1));
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = {mul2(v[i].re, d), mul2(v[i].im, d)};
  }
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) sts(at(pb, k1 + R1 * k2), swapped(v[slot<32>(k2)]));
  fence_async_shared();
  __syncthreads();
  if (here.leader()) {
    T::store_plane(&jobs.out[job], buf, x, kb);
    bulk_commit();
    bulk_wait_read_all();
  }
}

// The density's 3D spectrum [kx][ky][kz] from its (y, z)-transformed tiles, on request (not part of a solve).
template <int R1>
__global__ void __launch_bounds__(Cfg<R1>::Threads, Cfg<R1>::Blocks)
    fft_spectrum_kernel(const __grid_constant__ CUtensorMap in, const float2* __restrict__ tw, int blocks_kz,
                        float2* __restrict__ out, int* __restrict__ err) {
  using C = Cfg<R1>;
  extern __shared__ unsigned char raw[];
  __shared__ uint64_t bars[1];
  const Place<R1> here{raw, bars};
  const uint32_t buf = here.buf();
  const int ky = here.tile() / blocks_kz, kb = here.tile() - ky * blocks_kz;
  if (!fetch_tile(here, err, [&](uint32_t d, uint32_t b) { Tile<R1>::load_line(d, &in, ky, kb, b); })) return;
  const int lane = threadIdx.x & 31, warp = here.warp();
  const TileAddr at{buf, warp * C::P};
  C2 v[32];
#pragma unroll
  for (int p = 0; p < C::P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) v[p * R1 + m] = lds(at(p, lane + 32 * m));
  forward_lines<R1>(v, at, tw, lane);
  const int lb = C::second(lane), pb = lb / R1, k1 = lb % R1;
  const int kz = kb * 8 + 2 * (warp * C::P + pb), row = C::N / 2 + 1;
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) {
    const float2 re = unpack(v[slot<32>(k2)].re), im = unpack(v[slot<32>(k2)].im);
    float2* q = out + (static_cast<int64_t>(k1 + R1 * k2) * C::N + ky) * row + kz;
    if (kz < row) q[0] = make_float2(re.x, im.x);
    if (kz + 1 < row) q[1] = make_float2(re.y, im.y);
  }
}

// ---- x-pass -------------------------------------------------------------------------------------------------
// Learned factor of |k|, linearly interpolated, 1 beyond the table (without branches).
__device__ __forceinline__ float learned_factor(const FftSet& s, float kmag) {
  const float t = kmag * s.g_inv_dk;
  const int i = min(static_cast<int>(t), s.g_nk - 2);
  const float w = t - static_cast<float>(i);
  const float g = __ldg(s.g + i) * (1.f - w) + __ldg(s.g + i + 1) * w;
  return t >= static_cast<float>(s.g_nk - 1) ? 1.f : g;
}

struct XJobs {
  CUtensorMap in, out[4];
  FftSet set[2];
  int sets;
};

// One block per (ky, 8 kz) and filter set: forward along x, Green's function x filter x i, then inverse along x of the
// x component and of V.  Bound by issue and latency (three transforms on one tile's copies: 5000 instructions a warp;
// 3.15 ms at 1024^3 for 13.1 GB, 0.61 of the copy rate).  Between the two inverses the spectrum waits in registers
// (kKeep of a lane's 32 pairs) and in a stash beside the tile: with 255 registers a thread and 113 KB, two blocks of four
// warps per SM.  Other places for it were slower: made again by a second block (three blocks of 168 registers per SM)
// 3.77 ms, kept in the V spectrum's own lines in L2 3.85 ms.
constexpr int kKeep = 9;
// With a learned factor (MANY) a block holds as many tiles as give it four warps: they stay together at the block's barriers and
// share their instruction fetches, where blocks of one or two warps, at different places of a larger kernel, wait for theirs.
// Five fields, before and now: 512^3 4.01 -> 3.19 ms, 384^3 1.70 -> 1.46 ms, 256^3 508 -> 453 us; the plain kernels gain nothing
// by it (192^3 137 and 144 us).
template <int R1, bool MANY>
struct XCfg {
  static constexpr int G = MANY ? 4 / Cfg<R1>::W : 1;
  static constexpr int Threads = G * Cfg<R1>::Threads;
  static constexpr int Blocks = 8 / (Cfg<R1>::W * G);
  static constexpr int Stash = 32 - kKeep;
  static constexpr int Bytes = G * (Cfg<R1>::TileBytes + Cfg<R1>::W * Stash * 512) + 1024;
  // this warp's stash, behind the block's tiles
  __device__ __forceinline__ static uint32_t stash(uint32_t base) {
    return base + G * Cfg<R1>::TileBytes + (threadIdx.x >> 5) * (Stash * 512);
  }
};

template <int R1, bool LEARNED>
__global__ void __launch_bounds__(XCfg<R1, LEARNED>::Threads, XCfg<R1, LEARNED>::Blocks)
    fft_x_kernel(const __grid_constant__ XJobs jobs, const float2* __restrict__ tw, int blocks_kz, float kf, float scale,
                 int* __restrict__ err) {
  using C = Cfg<R1>;
  using T = Tile<R1>;
  constexpr int N = C::N, S = XCfg<R1, LEARNED>::Stash, G = XCfg<R1, LEARNED>::G;
  extern __shared__ unsigned char raw[];
  __shared__ uint64_t bars[G];
  const Place<R1, G> here{raw, bars};
  const uint32_t buf = here.buf();
  const unsigned tile = here.tile() / static_cast<unsigned>(jobs.sets);
  const int set = here.tile() - tile * jobs.sets;
  // 16 consecutive tiles share a region: ky mod 16 fastest
  const unsigned region = tile >> 4;
  const int kg = region / blocks_kz, kb = region - kg * blocks_kz, ky = kg * 16 + (tile & 15);
  if (!fetch_tile(here, err, [&](uint32_t d, uint32_t b) { T::load_line(d, &jobs.in, ky, kb, b); })) return;
  const int lane = threadIdx.x & 31, warp = here.warp();
  const TileAddr at{buf, warp * C::P};
  const uint32_t stash = XCfg<R1, LEARNED>::stash(here.base()) + lane * 16;
  const int lb = Cfg<R1>::second(lane), pb = lb / R1, k1 = lb % R1;
  C2 u[32], keep[kKeep];
  {
    C2 v[32];
#pragma unroll
    for (int p = 0; p < C::P; ++p)
#pragma unroll
      for (int m = 0; m < R1; ++m) v[p * R1 + m] = lds(at(p, lane + 32 * m));
    forward_lines<R1>(v, at, tw, lane);
    const FftSet& s = jobs.set[set];
    const int kz0 = kb * 8 + 2 * (warp * C::P + pb);
    const float kyf = kf * (ky < N / 2 ? ky : ky - N), kza = kf * kz0, kzb = kf * (kz0 + 1);
    const float k2a = kyf * kyf + kza * kza, k2b = kyf * kyf + kzb * kzb;
    const float wy = __ldg(s.wxy + ky);
    const float ca = wy * __ldg(s.wz + min(kz0, N / 2)), cb = wy * __ldg(s.wz + min(kz0 + 1, N / 2));
    const float* __restrict__ wx = s.wxy + k1;
    const u64 k2ab = pack(k2a, k2b), cab = pack(ca, cb), neg = both(-1.f);
    auto k_squared = [&](int k2, float kfx) {
      const int kx = k1 + R1 * k2;
      const u64 kxf = both(kfx * (k2 < 16 ? kx : kx - N));
      return fma2(kxf, kxf, k2ab);
    };
#pragma unroll
    for (int k2 = 0; k2 < 32; ++k2) {
      const float2 q = unpack(k_squared(k2, kf));
      const float fa = q.x > 0.f ? __fdividef(scale, q.x) : 0.f, fb = __fdividef(scale, q.y);
      const u64 c = mul2(pack(fa, fb), mul2(both(__ldg(wx + R1 * k2)), cab));
      // i c X with the parts swapped for the inverse: (c re, -c im)
      const C2 x = v[slot<32>(k2)];
      u[k2] = {mul2(x.re, c), mul2(x.im, mul2(c, neg))};
    }
    if (LEARNED && s.g != nullptr) {
      // |k|^2 again, hidden from the compiler, which else keeps all 64 of them from above
      float kfl = kf;
      asm volatile("" : "+f"(kfl));
#pragma unroll
      for (int k2 = 0; k2 < 32; ++k2) {
        const float2 q = unpack(k_squared(k2, kfl));
        const u64 g = pack(learned_factor(s, sqrtf(q.x)), learned_factor(s, sqrtf(q.y)));
        u[k2] = {mul2(u[k2].re, g), mul2(u[k2].im, g)};
      }
    }
  }
#pragma unroll
  for (int i = 0; i < S; ++i) sts(stash + i * 512, u[i]);
#pragma unroll
  for (int i = 0; i < kKeep; ++i) keep[i] = u[S + i];
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) {
    const u64 d = both(derivative(k1 + R1 * k2, N, kf));
    u[k2] = {mul2(u[k2].re, d), mul2(u[k2].im, d)};
  }
  inverse_first<R1>(u, tw, lane);
  inverse_second<R1>(u, at, lane);
  auto put = [&](int component) {
#pragma unroll
    for (int p = 0; p < C::P; ++p)
#pragma unroll
      for (int m = 0; m < R1; ++m) sts(at(p, lane + 32 * m), swapped(u[p * R1 + slot<R1>(m)]));
    fence_async_shared();
    __syncthreads();
    if (here.leader()) {
      T::store_line(&jobs.out[2 * set + component], buf, ky, kb);
      bulk_commit();
    }
  };
  put(0);
#pragma unroll
  for (int i = 0; i < S; ++i) u[i] = lds(stash + i * 512);
#pragma unroll
  for (int i = 0; i < kKeep; ++i) u[S + i] = keep[i];
  inverse_first<R1>(u, tw, lane);
  if (here.leader()) bulk_wait_read_all();  // the x component has left the tile
  __syncthreads();
  inverse_second<R1>(u, at, lane);
  put(1);
  if (here.leader()) bulk_wait_read_all();
}

// Transpose of the x-pass for one filter set: out = IFFT_x(-i c (d_x FFT_x(in[0]) + FFT_x(d_y in[1] + d_z in[2]))), the
// sum of the three cotangents' parts under the conjugate factors.  The first sum waits beside the tile, as in
// fft_x_kernel, while the x component comes into its place.
struct XAdjoint {
  CUtensorMap in[3], out;
  FftSet set;
};

template <int R1, bool LEARNED>
__global__ void __launch_bounds__(Cfg<R1>::Threads, XCfg<R1, false>::Blocks)
    fft_x_adjoint_kernel(const __grid_constant__ XAdjoint f, const float2* __restrict__ tw, int blocks_kz, float kf, float scale,
                         int* __restrict__ err) {
  using C = Cfg<R1>;
  using T = Tile<R1>;
  constexpr int N = C::N, S = XCfg<R1, false>::Stash;
  extern __shared__ unsigned char raw[];
  __shared__ uint64_t bars[1];
  const Place<R1> here{raw, bars};
  const uint32_t buf = here.buf();
  const unsigned region = here.tile() >> 4;
  const int kg = region / blocks_kz, kb = region - kg * blocks_kz, ky = kg * 16 + (here.tile() & 15);
  const int lane = threadIdx.x & 31, warp = here.warp();
  const TileAddr at{buf, warp * C::P};
  const uint32_t stash = XCfg<R1, false>::stash(here.base()) + lane * 16;
  const int lb = C::second(lane), pb = lb / R1, k1 = lb % R1;
  auto load = [&](const CUtensorMap* m) {
    return [=](uint32_t d, uint32_t b) { T::load_line(d, m, ky, kb, b); };
  };
  C2 v[32], keep[kKeep];
  if (!fetch_tile(here, err, load(&f.in[1]))) return;
  const u64 dy = both(derivative(ky, N, kf));
#pragma unroll
  for (int p = 0; p < C::P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const C2 x = lds(at(p, lane + 32 * m));
      v[p * R1 + m] = {mul2(x.re, dy), mul2(x.im, dy)};
    }
  if (!fetch_next(here, 1, err, load(&f.in[2]))) return;
#pragma unroll
  for (int p = 0; p < C::P; ++p) {
    const int kz = kb * 8 + 2 * (warp * C::P + p);
    const u64 dz = pack(kz == N / 2 ? 0.f : kf * kz, kf * (kz + 1));
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const C2 x = lds(at(p, lane + 32 * m));
      C2& y = v[p * R1 + m];
      y = {fma2(x.re, dz, y.re), fma2(x.im, dz, y.im)};
    }
  }
  forward_lines<R1>(v, at, tw, lane);
#pragma unroll
  for (int i = 0; i < S; ++i) sts(stash + i * 512, v[slot<32>(i)]);
#pragma unroll
  for (int i = 0; i < kKeep; ++i) keep[i] = v[slot<32>(S + i)];
  if (!fetch_next(here, 2, err, load(&f.in[0]))) return;
#pragma unroll
  for (int p = 0; p < C::P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) v[p * R1 + m] = lds(at(p, lane + 32 * m));
  forward_lines<R1>(v, at, tw, lane);
  C2 u[32];
  {
    const FftSet& s = f.set;
    const int kz0 = kb * 8 + 2 * (warp * C::P + pb);
    const float kyf = kf * (ky < N / 2 ? ky : ky - N), kza = kf * kz0, kzb = kf * (kz0 + 1);
    const float wy = __ldg(s.wxy + ky);
    const float ca = wy * __ldg(s.wz + min(kz0, N / 2)), cb = wy * __ldg(s.wz + min(kz0 + 1, N / 2));
    const float* __restrict__ wx = s.wxy + k1;
    const u64 k2ab = pack(kyf * kyf + kza * kza, kyf * kyf + kzb * kzb), cab = pack(ca, cb), neg = both(-1.f);
#pragma unroll
    for (int k2 = 0; k2 < 32; ++k2) {
      const int kx = k1 + R1 * k2;
      const u64 kxf = both(kf * (k2 < 16 ? kx : kx - N)), dx = both(derivative(kx, N, kf));
      const float2 q = unpack(fma2(kxf, kxf, k2ab));
      const float fa = q.x > 0.f ? __fdividef(scale, q.x) : 0.f, fb = __fdividef(scale, q.y);
      u64 c = mul2(pack(fa, fb), mul2(both(__ldg(wx + R1 * k2)), cab));
      if (LEARNED) c = mul2(c, pack(learned_factor(s, sqrtf(q.x)), learned_factor(s, sqrtf(q.y))));
      const C2 rest = k2 < S ? lds(stash + k2 * 512) : keep[k2 < S ? 0 : k2 - S], x = v[slot<32>(k2)];
      // -i c X with the parts swapped for the inverse: (-c re, c im)
      u[k2] = {mul2(fma2(x.re, dx, rest.re), mul2(c, neg)), mul2(fma2(x.im, dx, rest.im), c)};
    }
  }
  inverse_first<R1>(u, tw, lane);
  inverse_second<R1>(u, at, lane);
#pragma unroll
  for (int p = 0; p < C::P; ++p)
#pragma unroll
    for (int m = 0; m < R1; ++m) sts(at(p, lane + 32 * m), swapped(u[p * R1 + slot<R1>(m)]));
  fence_async_shared();
  __syncthreads();
  if (here.leader()) {
    T::store_line(&f.out, buf, ky, kb);
    bulk_commit();
    bulk_wait_read_all();
  }
}

// ---- launches -----------------------------------------------------------------------------------------------
template <class K>
hrt_status reserve(K kernel, int bytes) {
  return cuda_status(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes),
                     "shared memory of an FFT pass");
}

}  // namespace

template <int R1>
hrt_status Passes<R1>::forward(const FftPlan& p, float* rho, bool clear, cudaStream_t s) {
  using C = Cfg<R1>;
  const int kb = static_cast<int>(fft_row(C::N) / 8), smem = 4 * C::P * C::N * 16, groups = C::N * C::N / 4;
  HRT_TRY(reserve(fft_z_kernel<R1>, smem));
  fft_z_kernel<R1><<<groups / (4 * C::P), 128, smem, s>>>(ZForward{{rho}, {p.first}}, p.tw, groups,
                                                          2 * static_cast<int>(fft_row(C::N)), clear);
  HRT_LAUNCHED("fft_z_kernel");
  HRT_TRY(reserve(fft_y_kernel<R1>, C::TileBytes + 1024));
  fft_y_kernel<R1><<<C::N * kb, C::Threads, C::TileBytes + 1024, s>>>(YForward{{p.y_in}, {p.y_out}}, p.tw, kb, p.err);
  HRT_LAUNCHED("fft_y_kernel");
  return HRT_OK;
}

template <int R1>
hrt_status Passes<R1>::x_pass(const FftPlan& p, double box, double pref, const FftSet& a, const FftSet* b, cudaStream_t s) {
  using C = Cfg<R1>;
  const int kb = static_cast<int>(fft_row(C::N) / 8);
  XJobs j{};
  j.in = p.x_in;
  j.sets = b ? 2 : 1;
  for (int i = 0; i < 2 * j.sets; ++i) j.out[i] = p.x_out[i];
  j.set[0] = a;
  j.set[1] = b ? *b : a;
  const bool learned = a.g || (b && b->g);
  const auto kernel = learned ? fft_x_kernel<R1, true> : fft_x_kernel<R1, false>;
  using Many = XCfg<R1, true>;
  using One = XCfg<R1, false>;
  const int bytes = learned ? Many::Bytes : One::Bytes, threads = learned ? Many::Threads : One::Threads;
  const int blocks = C::N * kb * j.sets / (learned ? Many::G : One::G);
  HRT_TRY(reserve(kernel, bytes));
  const double scale = -pref / (static_cast<double>(C::N) * C::N * C::N);
  kernel<<<blocks, threads, bytes, s>>>(
      j, p.tw, kb, static_cast<float>(2.0 * M_PI / box), static_cast<float>(scale), p.err);
  HRT_LAUNCHED("fft_x_kernel");
  return HRT_OK;
}

template <int R1>
hrt_status Passes<R1>::inverse_y(const FftPlan& p, double box, bool rays, cudaStream_t s) {
  using C = Cfg<R1>;
  const int kb = static_cast<int>(fft_row(C::N) / 8);
  YJobs j{};
  j.jobs = rays ? 5 : 3;
  const int from[kFftMaxFields] = {0, 1, 1, 2, 3};
  for (int i = 0; i < j.jobs; ++i) {
    j.in[i] = p.iy_in[from[i]];
    j.out[i] = p.iy_out[i];
  }
  HRT_TRY(reserve(fft_iy_kernel<R1>, C::TileBytes + 1024));
  fft_iy_kernel<R1><<<C::N * kb * j.jobs, C::Threads, C::TileBytes + 1024, s>>>(
      j, p.tw, kb, static_cast<float>(2.0 * M_PI / box), p.err);
  HRT_LAUNCHED("fft_iy_kernel");
  return HRT_OK;
}

template <int R1>
hrt_status Passes<R1>::inverse_z(const FftPlan& p, float* grad, float* ray, cudaStream_t s) {
  using C = Cfg<R1>;
  const int smem = 4 * C::P * C::N * 16, groups = C::N * C::N / 4;
  const size_t cells = static_cast<size_t>(C::N) * C::N * C::N;
  ZFields f{};
  for (int i = 0; i < kFftMaxFields; ++i) {
    f.in[i] = p.out[i];
    f.out[i] = i < 3 ? grad + i * cells : ray ? ray + (i - 3) * cells : nullptr;
  }
  HRT_TRY(reserve(fft_iz_kernel<R1>, smem));
  fft_iz_kernel<R1><<<dim3(groups / (4 * C::P), ray ? 5 : 3), 128, smem, s>>>(f, p.tw, groups,
                                                                             2 * static_cast<int>(fft_row(C::N)));
  HRT_LAUNCHED("fft_iz_kernel");
  return HRT_OK;
}

template <int R1>
hrt_status Passes<R1>::adjoint(const FftPlan& p, double box, double pref, const FftSet& a, const float* grad_bar,
                               float* rho_bar, cudaStream_t s) {
  using C = Cfg<R1>;
  const FftAdjointPlan& q = p.adjoint;
  const int kb = static_cast<int>(fft_row(C::N) / 8), row = 2 * static_cast<int>(fft_row(C::N));
  const int zmem = 4 * C::P * C::N * 16, groups = C::N * C::N / 4, ymem = C::TileBytes + 1024;
  const size_t cells = static_cast<size_t>(C::N) * C::N * C::N;
  float* g = const_cast<float*>(grad_bar);  // read only: nothing is cleared
  HRT_TRY(reserve(fft_z_kernel<R1>, zmem));
  HRT_TRY(reserve(fft_y_kernel<R1>, ymem));
  // fields 0 and 1 together, then 2 through the first one's rows
  fft_z_kernel<R1><<<dim3(groups / (4 * C::P), 2), 128, zmem, s>>>(ZForward{{g, g + cells}, {q.rows[0], q.rows[1]}}, p.tw,
                                                                  groups, row, false);
  HRT_LAUNCHED("fft_z_kernel");
  fft_y_kernel<R1><<<dim3(C::N * kb, 2), C::Threads, ymem, s>>>(
      YForward{{q.y_in[0], q.y_in[1]}, {q.y_out[0], q.y_out[1]}}, p.tw, kb, p.err);
  HRT_LAUNCHED("fft_y_kernel");
  fft_z_kernel<R1><<<groups / (4 * C::P), 128, zmem, s>>>(ZForward{{g + 2 * cells}, {q.rows[0]}}, p.tw, groups, row, false);
  HRT_LAUNCHED("fft_z_kernel");
  fft_y_kernel<R1><<<C::N * kb, C::Threads, ymem, s>>>(YForward{{q.y_in[0]}, {q.y_out[2]}}, p.tw, kb, p.err);
  HRT_LAUNCHED("fft_y_kernel");
  XAdjoint x{{q.x_in[0], q.x_in[1], q.x_in[2]}, q.x_out, a};
  const auto kernel = a.g ? fft_x_adjoint_kernel<R1, true> : fft_x_adjoint_kernel<R1, false>;
  HRT_TRY(reserve(kernel, XCfg<R1, false>::Bytes));
  const float kf = static_cast<float>(2.0 * M_PI / box);
  kernel<<<C::N * kb, C::Threads, XCfg<R1, false>::Bytes, s>>>(
      x, p.tw, kb, kf, static_cast<float>(-pref / (static_cast<double>(C::N) * C::N * C::N)), p.err);
  HRT_LAUNCHED("fft_x_adjoint_kernel");
  YJobs y{};
  y.jobs = 1;
  y.in[0] = q.iy_in;
  y.out[0] = q.iy_out;
  HRT_TRY(reserve(fft_iy_kernel<R1>, ymem));
  fft_iy_kernel<R1><<<C::N * kb, C::Threads, ymem, s>>>(y, p.tw, kb, kf, p.err);
  HRT_LAUNCHED("fft_iy_kernel");
  ZFields z{};
  z.in[0] = q.rows[0];
  z.out[0] = rho_bar;
  HRT_TRY(reserve(fft_iz_kernel<R1>, zmem));
  fft_iz_kernel<R1><<<groups / (4 * C::P), 128, zmem, s>>>(z, p.tw, groups, row);
  HRT_LAUNCHED("fft_iz_kernel");
  return HRT_OK;
}

template <int R1>
hrt_status Passes<R1>::spectrum(const FftPlan& p, void* out, cudaStream_t s) {
  using C = Cfg<R1>;
  const int kb = static_cast<int>(fft_row(C::N) / 8);
  HRT_TRY(reserve(fft_spectrum_kernel<R1>, C::TileBytes + 1024));
  fft_spectrum_kernel<R1><<<C::N * kb, C::Threads, C::TileBytes + 1024, s>>>(p.x_in, p.tw, kb, static_cast<float2*>(out),
                                                                             p.err);
  HRT_LAUNCHED("fft_spectrum_kernel");
  return HRT_OK;
}

}  // namespace hrt
