// emd_fft.cuh -- declarations of the FFT form (csrc/emd_fft.cu), kept apart
// from emd_internal.cuh so that changes here leave the direct kernel's
// sources untouched.
#pragma once

#include "emd_internal.cuh"

namespace emd {

// FFT path: overlap-save on 128 x 128 tiles, two exposures per complex transform
struct FftLaunch {
  const float* x;       // current iterate (padded planes)
  float* xn;            // next iterate
  const float* N;       // numerator
  const float* u;       // n weight planes
  float2* w;            // weighted model images on the padded planes, as float2:
                        // Gaussian: plane q holds (w_2q, w_2q+1), each over its
                        // kernel's scale; Student-t: plane t holds (u'_t z_t, u'_t y_t)
  const float2* spec;   // pair spectra (fft_pair_spec float2 per pair and phase)
  const float2* spec1;  // Student-t: spectra of the single kernels
  const float* inv_scale;  // 1 / s_t of the pair spectra's kernels s_t k_t, powers of two;
                           // [n]: 0 if all are 1
  float2* scratch;      // r > 1, per (tile, group): the phases' x^, then the adjoint's
                        // accumulators
  const float* y;       // Student-t: n data planes (masked pixels 0)
  float nu;             // Student-t degrees of freedom; 0 = Gaussian
  int groups;           // exposure groups per tile (fft_groups)
  // groups > 1: accumulators of the groups of a tile, one slot per (tile, group), and
  // arrival counters per tile. Split launch (r = 1 Gaussian, at least
  // split_ctas tiles): one slot per CTA and a flag per tile (emd_fft.cu).
  float2* partials;
  int* counters;
  int split_ctas;       // SMs of the device
  int* err;  // device error word (a bounded wait that gives up sets kErrTimeout)
};

// The FFT buffer: byte offsets of its parts and its size. student: heavy-tailed
// noise; split_ctas: persistent CTAs of the split launch (0: none)
struct FftLayout {
  size_t spec, spec1, scale, w, scratch, partials, counters, total;
};
FftLayout fft_layout(const Shape& s, bool student, int split_ctas);
int fft_groups(const Shape& s);  // exposure groups per tile of this shape
size_t fft_smem_bytes();
int fft_tile_side(const Shape& s);
// inv_scale, spec (and, when not null, spec1) from the adjoint kernels ka
cudaError_t launch_fft_spectra(const Shape& s, const float* ka, float* inv_scale, float2* spec,
                               float2* spec1, cudaStream_t st);
cudaError_t launch_fft_iter(const Shape& s, const FftLaunch& a, cudaStream_t st);

// batch of FFT jobs: persistent forward and adjoint kernels over (job, tile and group)
struct FftBatchJob {
  Shape s;
  FftLaunch a[2];  // with x = buffer c, xn = buffer c^1, for c = cur
  int cur;
  int remaining;   // iterations still to run (0: skipped)
  int gxt;         // FFT tiles per row
};
int fft_tiles_x(const Shape& s);
int fft_tiles_total(const Shape& s);
cudaError_t launch_fft_batch(const FftBatchJob* jobs, int njobs, const int2* items,
                             const int* n_items, int* counters, int ctas, cudaStream_t st);

}  // namespace emd
