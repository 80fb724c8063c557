// emd_taps.cuh -- forms of the FP32 direct iteration whose passes are whole
// launches or grid-wide phases instead of a chain of tile items
// (declarations; the kernels are in emd_taps.cu).
#pragma once

#include "emd_internal.cuh"

namespace emd {

enum DirectForm {
  kFormHalo = 0,   // halo_kernel (emd_halo.cu)
  kFormTaps = 1,   // forward and adjoint launches, taps in the constant bank
  kFormSplit = 2   // one cooperative launch, (tile, exposure) items, grid barriers
};

// How a full FP32 direct iteration of this problem shape runs. Host only and
// independent of the device.
struct DirectPlan {
  int form;
  int tile;      // tile variant of the form
  int chunk;     // exposures per forward launch / phase
  int parts;     // 1: adjoint partials per exposure in work planes, summed in order
  int planes;    // work planes (the same for both noise models)
};
DirectPlan direct_plan(const Shape& s, bool student);

constexpr int kTapFloats = 7600;  // taps of one launch (30,400 bytes of kernel parameters)
// 16-byte aligned among the parameters, whatever comes before it: it is read as float4
struct alignas(16) TapBank {
  float k[kTapFloats];
};
static_assert(kTapFloats % 4 == 0, "the bank is read by quads");
// kernels (Kc x KP floats each) that one launch's constant bank holds
int tap_bank_kernels(const Shape& s);

struct DirectLaunch {
  FusedArgs a;      // x, xn, u, y, kf, ka, N, Nw, Den, err, nu
  float* work;      // plan.planes planes, zero outside the image
  int* counters;    // split: zero between launches (direct_counter_ints of them)
};
int direct_counter_ints(const Shape& s);

// One iteration with the taps form; hkf, hka: host copies of all kernels. Under stream
// capture the launches read h.a.kf and h.a.ka instead, so that a replay after a new
// frame set uses its PSFs.
cudaError_t launch_taps_iter(const Shape& s, const DirectPlan& p, const DirectLaunch& h,
                             const float* hkf, const float* hka, cudaStream_t st);
// iters iterations with the split form, x buffers xa (current) and xb
cudaError_t launch_split_iters(const Shape& s, const DirectPlan& p, const DirectLaunch& h,
                               float* xa, float* xb, int iters, cudaStream_t st);
// N = sum_t F_t^T (u_t y_t), where numerator_exposures(s) > 0 (the exposures whose
// kernels a launch can hold); hka: a host copy of the adjoint kernels; part: scratch,
// R2 planes each.
constexpr int kNumParts = 3;
int numerator_exposures(const Shape& s);
cudaError_t launch_numerator(const Shape& s, const float* u, const float* y, const float* hka,
                             float* N, float* const (&part)[kNumParts], cudaStream_t st);
// The log-likelihood's data term with the taps form: *nparts partial sums
// into part (at most max_parts, at least one per 64 x 64 tile), to be added in
// index order.
cudaError_t launch_taps_chi2(const Shape& s, const DirectPlan& p, const FusedArgs& a,
                             const float* hkf, double* part, int max_parts, int* nparts,
                             cudaStream_t st);
// iterations one split launch should run (a bound on its duration)
int split_iters_per_launch(const Shape& s);

}  // namespace emd
