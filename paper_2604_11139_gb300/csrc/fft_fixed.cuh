// complex128 FFT passes in 64-bit block fixed point (fft_fixed.cu).
//
// An FP64 instruction issues at 2 lanes per clock and SM on this chip, a 32-bit integer add or
// multiply at 64, so an FFT butterfly in FP64 runs 8 to 16 times slower than the same butterfly
// on 64-bit integers (an addition is two instructions, a product by a twiddle about seven).  The
// passes here read and write the same complex128 arrays as the FP64 kernels; inside a CTA each
// line's values are integers on one power-of-two scale taken from the line's largest input.
//
// Error: an input component is rounded to 2^-57 of its line's largest one (2^-56 at lengths from 120
// to 225, 2^-55 at 240 and 256), every product to one unit of the same scale and sums are exact,
// whatever the values' signs and sizes.  Components below 2^-4 (2^-3, 2^-2) of the largest thus enter
// with fewer bits than FP64 holds, as they would leave an FP64 transform: every output mixes the whole
// line.  The largest component is at most sqrt(n) times the r.m.s. of its line, so the error of a
// transform stays below that of one with FP64's 2^-53 rounding in every sum and product (measured on
// spectra from flat to a single component, tests/test_gpu_fixed_fft.py).  Subnormal components count
// as zero.
#pragma once
#include "pw_internal.cuh"

namespace pw {
namespace fx {

// Twiddles of one stage table entry w = exp(-2 pi i j m / L), as round(2^62 w) in signed 32-bit
// halves: value = hi 2^32 + lo with lo in (-2^31, 2^31).
struct Tw {
  int xlo, xhi, ylo, yhi;
};
static_assert(sizeof(Tw) == sizeof(double2), "the fixed-point table follows the FP64 one in memory");

// exp(-2 pi i k / L) for k < L, from long double sine and cosine.
std::vector<Tw> twiddles(int L);

// Whether the passes cover the box: every length with a two-stage plan, up to 256.
bool covers(const FftPlan& plan);

// The local part of the H-apply, as launch_local_apply<double>: out = kin psi + (V psi).
// tw: the plan's FP64 table, followed by the Tw table of the same layout at tw + plan.tw_total.
cudaError_t local_apply(const FftPlan& plan, const double2* tw, const SphereDev& sp, const double* vperm,
                        const double* kin, const double2* psi, int64_t ldpsi, int nband, double2* out, int64_t ldout,
                        double2* hb, int band_batch, cudaStream_t st, ::pw_ctx* prof);

// sum_b w_b Re[conj(a_b(r)) b_b(r)] added to the permuted grid, as launch_density<double> (b NULL: a).
// cudaErrorNotSupported before any launch when two x-lines and the sums exceed the shared memory.
cudaError_t density(const FftPlan& plan, const double2* tw, const SphereDev& sp, const double2* a, const double2* b,
                    int64_t ld, int nband, const double* w_dev, double* out_perm, double2* hb, int band_batch,
                    cudaStream_t st);

}  // namespace fx
}  // namespace pw
