// Host side of the FFT passes: tensor maps, twiddles and the choice of the side's kernels (fft_passes.cuh), of which the
// sides 256, 512 and 1024 are compiled here and the others in fft_passes_mid.cu and fft_passes_small.cu.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <vector>

#include "common.h"
#include "fft_passes.cuh"
#include "fft_passes.h"
#include "tma.h"

namespace hrt {

template struct Passes<8>;
template struct Passes<16>;
template struct Passes<32>;

namespace {

hrt_status encode(CUtensorMap* map, void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                  const cuuint32_t* box) {
  EncodeTiled enc = nullptr;
  HRT_TRY(tensor_map_encoder(&enc));
  const cuuint32_t one[5] = {1, 1, 1, 1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, rank, base, dims, strides, box, one,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(HRT_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", static_cast<int>(r));
  return HRT_OK;
}

// As Cfg::Rows.
cuuint32_t box_rows(int64_t n) { return static_cast<cuuint32_t>(n <= 256 ? n : n % 256 == 0 ? 256 : 128); }

// Rows [x][y][kz] as (floats of a row, rows), boxes of 8 kz x rows.
hrt_status plane_map(CUtensorMap* m, void* base, int64_t n) {
  const cuuint64_t row = 2 * fft_row(n), dims[2] = {row, static_cast<cuuint64_t>(n) * n}, strides[1] = {row * 4};
  const cuuint32_t box[2] = {16, box_rows(n)};
  return encode(m, base, 2, dims, strides, box);
}

// Tiles [ky / 16][kz / 8][x][ky mod 16][8 kz], boxes of all ky of an x (columns) or all x of a ky.
hrt_status tile_map(CUtensorMap* m, void* base, int64_t n, bool columns) {
  const cuuint64_t u = static_cast<cuuint64_t>(n), kb = fft_row(n) / 8;
  const cuuint64_t dims[5] = {16, 16, u, kb, u / 16}, strides[4] = {64, 1024, 1024 * u, 1024 * u * kb};
  const cuuint32_t rows = box_rows(n);
  const cuuint32_t column[5] = {16, 16, 1, 1, rows / 16}, line[5] = {16, 1, rows, 1, 1};
  return encode(m, base, 5, dims, strides, columns ? column : line);
}

}  // namespace

hrt_status tensor_map_encoder(EncodeTiled* out) {
  static std::once_flag once;
  static EncodeTiled fn = nullptr;
  static cudaError_t e = cudaSuccess;
  std::call_once(once, [] {
    cudaDriverEntryPointQueryResult q{};
    void* p = nullptr;
    e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
    if (e == cudaSuccess && q == cudaDriverEntryPointSuccess) fn = reinterpret_cast<EncodeTiled>(p);
  });
  if (!fn) return cuda_status(e == cudaSuccess ? cudaErrorSymbolNotFound : e, "cuTensorMapEncodeTiled entry point");
  *out = fn;
  return HRT_OK;
}

bool fft_supported(int64_t n) {
  switch (n) {
    case 64: case 96: case 128: case 192: case 256: case 384: case 512: case 768: case 1024: return true;
    default: return false;
  }
}

int64_t fft_row(int64_t n) { return (n / 2 + 1 + 7) / 8 * 8; }

size_t fft_spectrum_bytes(int64_t n) { return static_cast<size_t>(n) * n * fft_row(n) * 8; }

void fft_twiddles(int64_t n, std::vector<float2>& tw) {
  const int r1 = static_cast<int>(n / 32);
  tw.resize(static_cast<size_t>(r1) * 32 + 32 * 32);
  auto at = [n](int64_t l, int64_t k) {
    const double ph = 2.0 * M_PI * static_cast<double>((l * k) % n) / static_cast<double>(n);
    const float c = static_cast<float>(std::cos(ph)), s = static_cast<float>(std::sin(ph));
    return make_float2(c, s);
  };
  for (int k1 = 0; k1 < r1; ++k1)
    for (int l = 0; l < 32; ++l) tw[k1 * 32 + l] = at(l, k1);
  for (int n1 = 0; n1 < 32; ++n1)
    for (int t = 0; t < 32; ++t) tw[r1 * 32 + n1 * 32 + t] = at(n1, t % r1);
}

hrt_status fft_plan(FftPlan& p, int64_t n, int fields, void* half, void* const* mid, void* const* out,
                    const float2* tw, int* err) {
  p.n = n;
  p.fields = fields;
  p.tw = tw;
  p.err = err;
  p.first = static_cast<float*>(mid[0]);
  for (int i = 0; i < fields; ++i) p.out[i] = static_cast<float*>(out[i]);
  HRT_TRY(plane_map(&p.y_in, mid[0], n));
  HRT_TRY(tile_map(&p.y_out, half, n, true));
  HRT_TRY(tile_map(&p.x_in, half, n, false));
  for (int i = 0; i < (fields > 3 ? 4 : 2); ++i) {
    HRT_TRY(tile_map(&p.x_out[i], mid[i], n, false));
    HRT_TRY(tile_map(&p.iy_in[i], mid[i], n, true));
  }
  for (int i = 0; i < fields; ++i) HRT_TRY(plane_map(&p.iy_out[i], p.out[i], n));
  // the transposed solve: rows in mid[0] and mid[1]; tiles of the cotangents in the density's place and two fields'
  void* tiles[3] = {half, out[1], out[2]};
  FftAdjointPlan& a = p.adjoint;
  for (int i = 0; i < 2; ++i) {
    a.rows[i] = static_cast<float*>(mid[i]);
    HRT_TRY(plane_map(&a.y_in[i], mid[i], n));
  }
  for (int i = 0; i < 3; ++i) {
    HRT_TRY(tile_map(&a.y_out[i], tiles[i], n, true));
    HRT_TRY(tile_map(&a.x_in[i], tiles[i], n, false));
  }
  HRT_TRY(tile_map(&a.x_out, mid[1], n, false));
  HRT_TRY(tile_map(&a.iy_in, mid[1], n, true));
  return plane_map(&a.iy_out, mid[0], n);
}

#define HRT_FFT_SIDE(call)                                                           \
  switch (p.n) {                                                                     \
    case 64: return Passes<2>::call;                                                 \
    case 96: return Passes<3>::call;                                                 \
    case 128: return Passes<4>::call;                                                \
    case 192: return Passes<6>::call;                                                \
    case 256: return Passes<8>::call;                                                \
    case 384: return Passes<12>::call;                                               \
    case 512: return Passes<16>::call;                                               \
    case 768: return Passes<24>::call;                                               \
    case 1024: return Passes<32>::call;                                              \
    default: return fail(HRT_ERR_INVALID_ARG, "no FFT passes for this mesh side");   \
  }

hrt_status launch_fft_forward(const FftPlan& p, float* rho, bool clear, cudaStream_t s) {
  HRT_FFT_SIDE(forward(p, rho, clear, s))
}

hrt_status launch_fft_x(const FftPlan& p, double box, double pref, const FftSet& a, const FftSet* b, cudaStream_t s) {
  HRT_FFT_SIDE(x_pass(p, box, pref, a, b, s))
}

hrt_status launch_fft_inverse_y(const FftPlan& p, double box, bool rays, cudaStream_t s) {
  HRT_FFT_SIDE(inverse_y(p, box, rays, s))
}

hrt_status launch_fft_inverse_z(const FftPlan& p, float* grad, float* ray, cudaStream_t s) {
  HRT_FFT_SIDE(inverse_z(p, grad, ray, s))
}

hrt_status launch_fft_adjoint(const FftPlan& p, double box, double pref, const FftSet& a, const float* grad_bar, float* rho_bar,
                              cudaStream_t s) {
  HRT_FFT_SIDE(adjoint(p, box, pref, a, grad_bar, rho_bar, s))
}

hrt_status launch_fft_spectrum(const FftPlan& p, void* out, cudaStream_t s) { HRT_FFT_SIDE(spectrum(p, out, s)) }

}  // namespace hrt
