// emd_corr.cuh -- device code shared by the direct-form kernels (the fused
// CTA-pair kernel and the halo-exchange kernel): an FP64 block sum, and the
// register-blocked FP32 correlation, where a thread accumulates an RY x RX
// block of outputs
//     acc[p][c] += sum_{a < Kc, b < KP} k[a][b] src[oy + p + a][ox + c + b]
// from a shared-memory plane.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace emd {

// A staged plane whose rows carry a skew of 4 floats every RY rows, RY the
// row height of the reading threads' blocks: row R starts at
// base + R * pitch + 4 * (R / RY). With an even pitch the 8 lanes of a 16-byte
// load phase, RY rows apart, then fall on distinct bank groups.
struct SPlane {
  float* base;
  int pitch;
};

template <int RY>
__device__ __forceinline__ float* srow(const SPlane& p, int R) {
  return p.base + R * p.pitch + 4 * (R / RY);
}

template <int RX>
__device__ __forceinline__ void corr_window(float (&xv)[RX + 4], const float* row) {
#pragma unroll
  for (int m = 0; m < RX / 4 + 1; ++m) {
    const float4 v = reinterpret_cast<const float4*>(row)[m];
    xv[4 * m + 0] = v.x;
    xv[4 * m + 1] = v.y;
    xv[4 * m + 2] = v.z;
    xv[4 * m + 3] = v.w;
  }
}

// One output row takes one tap quad: one tap at a time across the outputs, so
// that consecutive FMAs share the tap's register and each accumulator takes
// its taps in order.
template <int RX>
__device__ __forceinline__ void corr_taps(float (&acc)[RX], const float4 k,
                                          const float (&xv)[RX + 4]) {
#pragma unroll
  for (int c = 0; c < RX; ++c) acc[c] = fmaf(k.x, xv[c + 0], acc[c]);
#pragma unroll
  for (int c = 0; c < RX; ++c) acc[c] = fmaf(k.y, xv[c + 1], acc[c]);
#pragma unroll
  for (int c = 0; c < RX; ++c) acc[c] = fmaf(k.z, xv[c + 2], acc[c]);
#pragma unroll
  for (int c = 0; c < RX; ++c) acc[c] = fmaf(k.w, xv[c + 3], acc[c]);
}

template <int RY, int RX>
__device__ __forceinline__ void corr_zero(float (&a)[RY][RX]) {
#pragma unroll
  for (int p = 0; p < RY; ++p)
#pragma unroll
    for (int c = 0; c < RX; ++c) a[p][c] = 0.f;
}
template <int RY, int RX>
__device__ __forceinline__ void corr_add(float (&sum)[RY][RX], const float (&a)[RY][RX]) {
#pragma unroll
  for (int p = 0; p < RY; ++p)
#pragma unroll
    for (int c = 0; c < RX; ++c) sum[p][c] += a[p][c];
}
// where a correlation's FMAs go: the block sums where there are any, else the sums
template <int RY, int RX>
__device__ __forceinline__ float (&corr_target(float (&)[RY][RX], float (&block)[RY][RX]))[RY][RX] {
  return block;
}
template <int RY, int RX>
__device__ __forceinline__ float (&corr_target(float (&sum)[RY][RX], float (&)[1][1]))[RY][RX] {
  return sum;
}

// U source rows (U = 2 or 4) of a block of four output rows, the first at row
// s: xb[0] holds its window, q[j] the quad of kernel row s - 1 - j; skew: 4 if
// s mod 4 = 3 (the rows' skew steps at the next row), else 0. The next row's
// window is loaded before a row's FMAs. On return xb[0] holds row s + U.
template <int U, int RX>
__device__ __forceinline__ void corr4_rows(float (&acc)[4][RX], float4 (&q)[3],
                                           float (&xb)[2][RX + 4], const float*& row,
                                           const float*& kq, int pitch, int KP, int skew) {
  float4 nw[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    nw[u] = *reinterpret_cast<const float4*>(kq);
    kq += KP;
    row += u == 0 ? pitch + skew : pitch;
    corr_window<RX>(xb[(u + 1) & 1], row);
#pragma unroll
    for (int p = 0; p < 4; ++p) corr_taps<RX>(acc[p], p <= u ? nw[u - p] : q[p - u - 1], xb[u & 1]);
  }
  if (U == 2) q[2] = q[0];
#pragma unroll
  for (int j = 0; j < (U == 2 ? 2 : 3); ++j) q[j] = nw[U - 1 - j];
}

// U source rows of a block of three output rows, the first at row s = 2 mod 3 (or a
// later one of its three, skew 0): q[j] the quad of kernel row s - 1 - j.
template <int U, int RX>
__device__ __forceinline__ void corr3_rows(float (&acc)[3][RX], float4 (&q)[2], const float*& row,
                                           const float*& kq, int pitch, int KP, int skew) {
  float4 nw[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    float xv[RX + 4];
    corr_window<RX>(xv, row);
    nw[u] = *reinterpret_cast<const float4*>(kq);
    kq += KP;
    row += u == 0 ? pitch + skew : pitch;
#pragma unroll
    for (int p = 0; p < 3; ++p) corr_taps<RX>(acc[p], p <= u ? nw[u - p] : q[p - u - 1], xv);
  }
  q[1] = U == 1 ? q[0] : nw[U == 1 ? 0 : U - 2];
  q[0] = nw[U - 1];
}

// The loop that bounds every direct-form kernel, on blocks of RY x RX outputs
// (oy a multiple of RY; Kc odd). Tap quads outside, source rows inside: a
// quad that a source row brings for output row 0 stays in a register for
// output row 1 at the next source row. Every output sums its taps in the
// same order (quads ascending, in a quad rows ascending, in a row columns
// ascending) whatever block it falls in.
//
// RY = 2, 16 warps an SM: 62 TFLOP/s at K = 43 on a 64 x 128 tile (loop
// alone, 80.5 derived peak). The same loop on 4 x 16 blocks, 8 warps an SM,
// reaches 52-58 however it is unrolled or prefetched, rows outside and quads
// inside 55: all execute over 90 % FMAs, and what differs is the dispatch
// stall (0.3-0.5 per issue), which more warps cover and a larger block, with
// fewer loads, does not.
//
// BLOCKS (the numerator): the taps of each quad of columns are summed from zero
// and the blocks then added. One FP32 chain of Kc^2 terms would leave an error
// that no later iteration takes out again, since N is computed once per frame set;
// blocks of 4 Kc leave about half of it (43 x 43, 2e-7 -> 9e-8).
//
// CHECKED (halo_kernel's 64-row tiles): the loop with its edges checked inside instead
// of the unrolled triangles. No quad moves between
// registers: 5 x 4096^2, K = 43: 12.73 -> 12.41 ms, K = 25, 12 x 2048^2: 3.47 -> 3.27 (one image of
// few tiles, where a chain of items sets the time, 16 x 900^2, K = 43: 2.98 -> 3.18).
template <int RY, int RX, bool BLOCKS = false, bool CHECKED = false>
__device__ __forceinline__ void corr_tile(float (&sum)[RY][RX], const SPlane& src, int oy,
                                          int ox, const float* __restrict__ ks, int KP,
                                          int Kc) {
  static_assert(!BLOCKS || RY == 2, "blocks are summed in the two-row form only");
  const float* col = srow<RY>(src, oy) + ox;
  const int pitch = src.pitch;
  float block[BLOCKS ? RY : 1][BLOCKS ? RX : 1];
  float(&acc)[RY][RX] = corr_target<RY, RX>(sum, block);
  if constexpr (RY == 2) {
#pragma unroll 1
    for (int b = 0; b < KP; b += 4) {
      if (BLOCKS) corr_zero<RY, RX>(acc);
      const float* row = col + b;  // row s at row + s * pitch + 4 * (s / 2)
      const float* kq = ks + b;
      float xv[RX + 4];
      // source row 0: output row 0 only
      corr_window<RX>(xv, row);
      float4 k1 = *reinterpret_cast<const float4*>(kq);  // the quad of the row before
      corr_taps<RX>(acc[0], k1, xv);
      row += pitch;
      kq += KP;
      corr_window<RX>(xv, row);
#pragma unroll 1
      for (int s = 1; s < Kc; s += 2) {  // rows s and s + 1 (Kc - 1 is even)
        const float4 ka = *reinterpret_cast<const float4*>(kq);
        corr_taps<RX>(acc[0], ka, xv);
        corr_taps<RX>(acc[1], k1, xv);
        row += pitch + 4;
        corr_window<RX>(xv, row);
        k1 = *reinterpret_cast<const float4*>(kq + KP);
        corr_taps<RX>(acc[0], k1, xv);
        corr_taps<RX>(acc[1], ka, xv);
        row += pitch;
        kq += 2 * KP;
        corr_window<RX>(xv, row);
      }
      corr_taps<RX>(acc[1], k1, xv);  // source row Kc: output row 1 only
      if (BLOCKS) corr_add<RY, RX>(sum, acc);
    }
    return;
  }
  if constexpr (RY == 3) {
    // rows 0, 1 and Kc, Kc + 1 as unrolled triangles, three rows at a time between
    // (edges checked inside the loop: 16 x 900^2, K = 43: 3.22 ms, 2.81 here)
    if (Kc >= 3) {
#pragma unroll 1
      for (int b = 0; b < KP; b += 4) {
        const float* row = col + b;  // row s at row + s * pitch + 4 * (s / 3)
        const float* kq = ks + b;
        float xv[RX + 4];
        float4 q[2];
        corr_window<RX>(xv, row);
        q[1] = *reinterpret_cast<const float4*>(kq);
        corr_taps<RX>(acc[0], q[1], xv);
        row += pitch;
        corr_window<RX>(xv, row);
        q[0] = *reinterpret_cast<const float4*>(kq + KP);
        corr_taps<RX>(acc[0], q[0], xv);
        corr_taps<RX>(acc[1], q[1], xv);
        row += pitch;
        kq += 2 * KP;
        int s = 2;
#pragma unroll 1
        for (; s + 3 <= Kc; s += 3) corr3_rows<3, RX>(acc, q, row, kq, pitch, KP, 4);
#pragma unroll 1
        for (int skew = 4; s < Kc; ++s, skew = 0)
          corr3_rows<1, RX>(acc, q, row, kq, pitch, KP, skew);
        corr_window<RX>(xv, row);
        corr_taps<RX>(acc[1], q[0], xv);
        corr_taps<RX>(acc[2], q[1], xv);
        row += Kc % 3 == 2 ? pitch + 4 : pitch;
        corr_window<RX>(xv, row);
        corr_taps<RX>(acc[2], q[0], xv);
      }
      return;
    }
  }
  if constexpr (RY == 4 && !CHECKED) {
    // rows 0 .. 2 and Kc .. Kc + 2 as unrolled triangles, no checks between
    if (Kc >= 3) {
#pragma unroll 1
      for (int b = 0; b < KP; b += 4) {
        const float* row = col + b;
        const float* kq = ks + b;
        float xb[2][RX + 4];
        float4 q[3];
        corr_window<RX>(xb[0], row);
        q[2] = *reinterpret_cast<const float4*>(kq);
        q[1] = *reinterpret_cast<const float4*>(kq + KP);
        q[0] = *reinterpret_cast<const float4*>(kq + 2 * KP);
        kq += 3 * KP;
        row += pitch;
        corr_window<RX>(xb[1], row);
        corr_taps<RX>(acc[0], q[2], xb[0]);
        row += pitch;
        corr_window<RX>(xb[0], row);
        corr_taps<RX>(acc[0], q[1], xb[1]);
        corr_taps<RX>(acc[1], q[2], xb[1]);
        row += pitch;
        corr_window<RX>(xb[1], row);
        corr_taps<RX>(acc[0], q[0], xb[0]);
        corr_taps<RX>(acc[1], q[1], xb[0]);
        corr_taps<RX>(acc[2], q[2], xb[0]);
#pragma unroll
        for (int c = 0; c < RX + 4; ++c) xb[0][c] = xb[1][c];
        // Kc mod 4 = 1: two rows at a time, one loop: a remainder after the
        // four-row loop would push the code out of the instruction cache
        if ((Kc & 3) == 3) {
#pragma unroll 1
          for (int s = 3; s < Kc; s += 4) corr4_rows<4, RX>(acc, q, xb, row, kq, pitch, KP, 4);
        } else {
#pragma unroll 1
          for (int s = 3, skew = 4; s < Kc; s += 2, skew ^= 4)
            corr4_rows<2, RX>(acc, q, xb, row, kq, pitch, KP, skew);
        }
        row += (Kc & 3) == 3 ? pitch + 4 : pitch;
        corr_window<RX>(xb[1], row);
        corr_taps<RX>(acc[1], q[0], xb[0]);
        corr_taps<RX>(acc[2], q[1], xb[0]);
        corr_taps<RX>(acc[3], q[2], xb[0]);
        row += pitch;
        corr_window<RX>(xb[0], row);
        corr_taps<RX>(acc[2], q[0], xb[1]);
        corr_taps<RX>(acc[3], q[1], xb[1]);
        corr_taps<RX>(acc[3], q[0], xb[0]);
      }
      return;
    }
  }
#pragma unroll 1
  for (int b = 0; b < KP; b += 4) {
    float4 kv[RY];  // quad of kernel row a in slot a mod RY
    const float* row = col + b;
    const float* kq = ks + b;
#pragma unroll 1
    for (int s0 = 0; s0 < Kc + RY - 1; s0 += RY, row += RY * pitch + 4, kq += RY * KP) {
#pragma unroll
      for (int u = 0; u < RY; ++u) {
        const int s = s0 + u;
        if (s >= Kc + RY - 1) break;
        float xv[RX + 4];
        corr_window<RX>(xv, row + u * pitch);
        if (s < Kc) kv[u] = *reinterpret_cast<const float4*>(kq + u * KP);
#pragma unroll
        for (int p = 0; p < RY; ++p)
          if (s - p >= 0 && s - p < Kc) corr_taps<RX>(acc[p], kv[(u + RY - p) % RY], xv);
      }
    }
  }
}

// Stages the window of `rows` rows and `cols` columns (a multiple of 4) whose
// first row is at `base` (a row start of a padded plane, 16-byte aligned; pitch
// P a multiple of 4) and whose first column is c0. Four staged columns are
// one 16-byte shared store, cut from the two 16-byte words of the plane's
// grid that they straddle (the second word is the neighbour's first, an L1
// hit): four scalar stores per word would conflict four ways. LOADS words
// in flight per thread. CG: loads bypass L1 (the plane is written by other
// SMs during the launch). stage_words: the words come from load(offset from the
// row start `base` would be).
template <int RY, int NT, int LOADS, class Load>
__device__ __forceinline__ void stage_words(const SPlane& sp, Load&& load, int P, int c0, int rows,
                                            int cols) {
  const int sh = c0 & 3, nq = cols >> 2;
  const int total = rows * nq;
  for (int e0 = threadIdx.x; e0 < total; e0 += NT * LOADS) {
    float4 v[LOADS], w[LOADS];
#pragma unroll
    for (int q = 0; q < LOADS; ++q) {
      const int e = e0 + q * NT;
      if (e < total) {
        const int R = e / nq, m = e - R * nq;
        const long long off = (long long)R * P + (c0 & ~3) + 4 * m;
        v[q] = load(off);
        if (sh) w[q] = load(off + 4);
      }
    }
#pragma unroll
    for (int q = 0; q < LOADS; ++q) {
      const int e = e0 + q * NT;
      if (e < total) {
        const int R = e / nq, m = e - R * nq;
        float4 o = v[q];
        if (sh == 1) o = make_float4(v[q].y, v[q].z, v[q].w, w[q].x);
        if (sh == 2) o = make_float4(v[q].z, v[q].w, w[q].x, w[q].y);
        if (sh == 3) o = make_float4(v[q].w, w[q].x, w[q].y, w[q].z);
        reinterpret_cast<float4*>(srow<RY>(sp, R))[m] = o;
      }
    }
  }
}

template <int RY, int NT, int LOADS, bool CG>
__device__ __forceinline__ void stage_window(const SPlane& sp, const float* base, int P, int c0,
                                             int rows, int cols) {
  stage_words<RY, NT, LOADS>(
      sp,
      [base](long long off) {
        const float4* p = reinterpret_cast<const float4*>(base + off);
        return CG ? __ldcg(p) : __ldg(p);
      },
      P, c0, rows, cols);
}

// flags between CTAs
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ int ld_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

constexpr uint32_t kBarrierPolls = 1u << 23;  // x ~0.5 us per poll: seconds, not a hang

// Grid barrier number `round` (from 1) of a cooperative launch; every thread
// of the CTA calls it. Bounded: a wait that gives up raises the abort flag,
// which ends all later waits; returns false then. ctrl: [0] arrivals, [1] CTAs
// finished, [2] abort flag.
__device__ __forceinline__ bool grid_barrier(int* ctrl, int round, int* ok_s) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(&ctrl[0], 1);
    const int target = round * (int)gridDim.x;
    uint32_t i = 0;
    bool ok = false;
    for (; i < kBarrierPolls; ++i) {
      if (ld_acquire(&ctrl[0]) >= target) {
        ok = true;
        break;
      }
      if (ld_relaxed(&ctrl[2])) break;
      if (i > 64) __nanosleep(100);
    }
    if (!ok) atomicExch(&ctrl[2], 1);
    *ok_s = ok;
  }
  __syncthreads();
  return *ok_s != 0;
}

// Sum of v over the CTA, in FP64 (warp shuffles, then the warps in order).
__device__ __forceinline__ double block_sum_f64(double v, double* red /* >= 8 */) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  return s;  // valid in thread 0
}

}  // namespace emd
