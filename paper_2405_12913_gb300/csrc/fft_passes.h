// The passes of the split Poisson solve (fft_passes.cu): real-to-complex FFT along z, FFTs along y, one pass along x
// that holds the k-space step, inverse FFTs along y and complex-to-real FFTs along z.  Every 3D spectrum crosses
// memory once per pass, in layouts of the passes' own.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "common.h"

namespace hrt {

// Mesh sides the passes support: 64, 96, 128, 192, 256, 384, 512, 768, 1024.
bool fft_supported(int64_t n);
// kz columns of a row, n/2 + 1 rounded up to the 8 of a tile.
int64_t fft_row(int64_t n);
// Bytes of one spectrum in either layout.
size_t fft_spectrum_bytes(int64_t n);
// Bit a pass sets in its error word when a wait for a tile's copy timed out (its block then stops).
constexpr int kFftTimeout = 1;
constexpr int kFftMaxFields = 5;
// Twiddles as the passes read them, (cos, sin) of 2 pi l k1 / n at [k1][l] then the same at [n1][lane] for the
// inverse along a lane's k1; FP64 on the host, rounded to float.
void fft_twiddles(int64_t n, std::vector<float2>& tw);

// One filter set: per-axis factor tables wxy [n] (signed-frequency order) and wz [n/2 + 1] and the optional learned
// factor g(|k|) (g_nk entries over [0, (g_nk - 1) / g_inv_dk]).
struct FftSet {
  const float* wxy;
  const float* wz;
  const float* g;
  int g_nk;
  float g_inv_dk;
};

// Tensor maps of the transposed solve, over the plan's five (or more) spectra: two for rows, three for tiles.
struct FftAdjointPlan {
  float* rows[2] = {};
  CUtensorMap y_in[2], y_out[3], x_in[3], x_out, iy_in, iy_out;
};

// Device buffers of one mesh size and the tensor maps over them.  half holds the (y, z)-transformed density (and,
// once the x-pass has read it, the first field of the inverse y-pass); mid the outputs of the x-pass, an x component
// and V per filter set; out[j] field j between the inverse y- and z-passes (out[0] is half).
struct FftPlan {
  int64_t n = 0;
  int fields = 0;  // 3, or 5 with ray fields
  const float2* tw = nullptr;
  int* err = nullptr;
  float* out[kFftMaxFields] = {};
  float* first = nullptr;  // output of the forward z-pass (mid[0])
  CUtensorMap y_in, y_out, x_in, x_out[4], iy_in[4], iy_out[kFftMaxFields];
  FftAdjointPlan adjoint;
};

// Fills the plan's maps; half, mid[2 or 4] and out[fields] are spectra of fft_spectrum_bytes(n), 128-byte aligned.  out[0]
// may be half where its spectrum is not asked for after a solve.
hrt_status fft_plan(FftPlan& p, int64_t n, int fields, void* half, void* const* mid, void* const* out,
                    const float2* tw, int* err);
// rho -> (y, z)-transformed density; clear: rho is set to zero once it has been read.
hrt_status launch_fft_forward(const FftPlan& p, float* rho, bool clear, cudaStream_t s);
// The x-pass: with set b (nullptr: none) for the ray fields.
hrt_status launch_fft_x(const FftPlan& p, double box, double pref, const FftSet& a, const FftSet* b, cudaStream_t s);
// grad [3][n^3], and ray [2][n^3] (or nullptr).
hrt_status launch_fft_inverse_y(const FftPlan& p, double box, bool rays, cudaStream_t s);
hrt_status launch_fft_inverse_z(const FftPlan& p, float* grad, float* ray, cudaStream_t s);
// rho_bar [n^3] from the cotangents grad_bar [3][n^3] of the fields of one filter set (hrt_pm_solve_adjoint); overwrites
// the plan's spectra.
hrt_status launch_fft_adjoint(const FftPlan& p, double box, double pref, const FftSet& a, const float* grad_bar, float* rho_bar,
                              cudaStream_t s);
// The 3D half spectrum [kx][ky][kz] (complex64) of the density last given to launch_fft_forward; half must still hold it
// (out[0] is a buffer of its own).
hrt_status launch_fft_spectrum(const FftPlan& p, void* out, cudaStream_t s);

// The launches for side 32 R1 (fft_passes.cuh).
template <int R1>
struct Passes {
  static hrt_status forward(const FftPlan& p, float* rho, bool clear, cudaStream_t s);
  static hrt_status x_pass(const FftPlan& p, double box, double pref, const FftSet& a, const FftSet* b, cudaStream_t s);
  static hrt_status inverse_y(const FftPlan& p, double box, bool rays, cudaStream_t s);
  static hrt_status inverse_z(const FftPlan& p, float* grad, float* ray, cudaStream_t s);
  static hrt_status adjoint(const FftPlan& p, double box, double pref, const FftSet& a, const float* grad_bar, float* rho_bar,
                            cudaStream_t s);
  static hrt_status spectrum(const FftPlan& p, void* out, cudaStream_t s);
};
extern template struct Passes<2>;
extern template struct Passes<3>;
extern template struct Passes<4>;
extern template struct Passes<6>;
extern template struct Passes<12>;
extern template struct Passes<24>;

}  // namespace hrt
