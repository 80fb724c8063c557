// emd_taps.cu -- the FP32 direct EM iteration of Sec. 2, Eq. (2) (Eq. (3) for
// r > 1) without a chain of tile items: per chunk of exposures a forward pass
// (w_t = u_t . F_t x into work planes) and an adjoint pass (Den += F_t^T w_t,
// the last chunk applying the update), in two forms.
//
// Taps form (large frame sets). Each pass is a launch that carries the taps
// of its chunk's kernels in its parameters, so the correlation loop reads them
// from the constant bank instead of shared memory: they never pass through
// the vector registers, and the loop runs at 68-72 TFLOP/s of the derived
// 80.5 (K = 43, 64 x 128 tiles), against 55 with the taps in shared memory,
// whose limit is the dispatch stall of FMAs with three register operands.
// 30 KB of parameters hold 4 kernels of 43 x 43. Large images add each
// exposure to Den as it is done; smaller ones keep a chunk's sums in work
// planes and a third launch adds them in exposure order, so that exposures run
// side by side. 4096^2 x 33, K = 43: 78.8 ms an iteration in halo_kernel,
// 62.8 here (0.81 of the derived FP32 peak); bound by the FMA pipe, 44 taps a
// row for 43, and each launch's last wave.
//
// Split form (images of a few tiles). halo_kernel adds the exposures of a
// tile one after the other, so a 128 x 128 image keeps 2 of 152 SMs busy. Here
// (tile, exposure) items are independent: every exposure's adjoint sum goes
// to a work plane of its own and the last CTA to finish a tile adds the planes
// in exposure order. One cooperative launch runs many iterations, two
// grid barriers each; tiles of 32 x 64, or 32 x 32 for small images. Bound by barriers
// and latency
// (128 x 128 x 4, K = 15: 104 -> 29 us an iteration).
//
// Both give halo_kernel's iterates bit for bit: every output's taps are
// summed in the same order (emd_corr.cuh), each exposure's adjoint sum starts
// at zero, and the sums are added in exposure order.
#include <algorithm>
#include <type_traits>

#include "emd_corr.cuh"
#include "emd_taps.cuh"

namespace emd {

namespace {

constexpr int kSMs = 152;

// ---------------------------------------------------------------------------
// correlation with the taps in the constant bank
// ---------------------------------------------------------------------------

__device__ __forceinline__ float4 bank_quad(const TapBank& bank, int off) {
  return reinterpret_cast<const float4*>(bank.k)[off >> 2];
}

// U source rows (U = 2 or 4), the first at row s: xv holds its window, q[j] the
// quad of kernel row s - 1 - j; skew: 4 if s mod 4 = 3 (the rows' skew steps at
// the next row), else 0. On return xv holds row s + U.
template <int U>
__device__ __forceinline__ void bank_rows(float (&acc)[4][16], float4 (&q)[3], float (&xv)[20],
                                          const float*& row, int& ko, int pitch, int KP,
                                          const TapBank& bank, int skew) {
  float4 nw[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    nw[u] = bank_quad(bank, ko);
    ko += KP;
    row += u == 0 ? pitch + skew : pitch;
#pragma unroll
    for (int p = 0; p < 4; ++p) corr_taps<16>(acc[p], p <= u ? nw[u - p] : q[p - u - 1], xv);
    corr_window<16>(xv, row);
  }
  if (U == 2) q[2] = q[0];
#pragma unroll
  for (int j = 0; j < (U == 2 ? 2 : 3); ++j) q[j] = nw[U - 1 - j];
}

// corr_tile<4, 16> with the kernel at bank.k[koff ..] (Kc odd and >= 5, rows
// of KP floats): the same sums in the same order, in blocks (corr_tile) too. Rows 0 .. 2 and Kc .. Kc + 2
// are unrolled triangles, so the loop over the rows between carries no checks.
template <bool BLOCKS = false>
__device__ __forceinline__ void corr_bank(float (&sum)[4][16], const SPlane& src, int oy, int ox,
                                          const TapBank& bank, int koff, int KP, int Kc) {
  const float* col = srow<4>(src, oy) + ox;
  const int pitch = src.pitch;
  float block[BLOCKS ? 4 : 1][BLOCKS ? 16 : 1];
  float(&acc)[4][16] = corr_target<4, 16>(sum, block);
#pragma unroll 1
  for (int b = 0; b < KP; b += 4) {
    if (BLOCKS) corr_zero<4, 16>(acc);
    const float* row = col + b;
    int ko = koff + b;
    float xv[20];
    float4 q[3];
    corr_window<16>(xv, row);
    const float4 k0 = bank_quad(bank, ko), k1 = bank_quad(bank, ko + KP),
                 k2 = bank_quad(bank, ko + 2 * KP);
    ko += 3 * KP;
    corr_taps<16>(acc[0], k0, xv);
    row += pitch;
    corr_window<16>(xv, row);
    corr_taps<16>(acc[0], k1, xv);
    corr_taps<16>(acc[1], k0, xv);
    row += pitch;
    corr_window<16>(xv, row);
    corr_taps<16>(acc[0], k2, xv);
    corr_taps<16>(acc[1], k1, xv);
    corr_taps<16>(acc[2], k0, xv);
    row += pitch;
    corr_window<16>(xv, row);
    q[0] = k2;
    q[1] = k1;
    q[2] = k0;
    // Kc mod 4 = 1: two rows at a time, one loop: a remainder after the
    // four-row loop pushed the code out of the instruction cache (K = 25 at 40
    // TFLOP/s)
    if ((Kc & 3) == 3) {
#pragma unroll 1
      for (int s = 3; s < Kc; s += 4) bank_rows<4>(acc, q, xv, row, ko, pitch, KP, bank, 4);
    } else {
#pragma unroll 1
      for (int s = 3, skew = 4; s < Kc; s += 2, skew ^= 4)
        bank_rows<2>(acc, q, xv, row, ko, pitch, KP, bank, skew);
    }
    corr_taps<16>(acc[1], q[0], xv);
    corr_taps<16>(acc[2], q[1], xv);
    corr_taps<16>(acc[3], q[2], xv);
    row += (Kc & 3) == 3 ? pitch + 4 : pitch;
    corr_window<16>(xv, row);
    corr_taps<16>(acc[2], q[0], xv);
    corr_taps<16>(acc[3], q[1], xv);
    row += pitch;
    corr_window<16>(xv, row);
    corr_taps<16>(acc[3], q[0], xv);
    if (BLOCKS) corr_add<4, 16>(sum, acc);
  }
}

// Where a launch's taps are: in its parameters (TapBank), or, for a launch that is
// captured into a graph, in the context's arena (TapMemory), because a graph keeps
// the parameters of its capture and would replay the PSFs of that time after a new
// frame set. The kernel's taps then pass through shared memory (ks), as in
// halo_kernel, and the loop runs at its rate (corr_tile; the same bits).
struct TapMemory {
  const float* k;
};

template <int NT>
__device__ __forceinline__ void corr_launch(float (&acc)[4][16], const SPlane& src, int oy, int ox,
                                            const TapBank& bank, int koff, int KP, int Kc, float*) {
  corr_bank(acc, src, oy, ox, bank, koff, KP, Kc);
}
template <int NT>
__device__ __forceinline__ void corr_launch(float (&acc)[4][16], const SPlane& src, int oy, int ox,
                                            const TapMemory& mem, int koff, int KP, int Kc,
                                            float* ks) {
  __syncthreads();  // readers of the previous kernel are done
  for (int q = threadIdx.x; q < (Kc * KP) >> 2; q += NT)
    reinterpret_cast<float4*>(ks)[q] = __ldg(reinterpret_cast<const float4*>(mem.k + koff) + q);
  __syncthreads();
  corr_tile<4, 16>(acc, src, oy, ox, ks, KP, Kc);
}

// ---------------------------------------------------------------------------
// pieces shared by both forms; a thread's block: RY x RX outputs at image
// rows i .., columns j ..
// ---------------------------------------------------------------------------

__device__ __forceinline__ float student_weight(float u, float y, float z, float nu) {
  const float d = y - z;
  return u > 0.f ? u * (nu + 1.f) / fmaf(u * d, d, nu) : 0.f;
}

// w = u z (heavy-tailed: w = u' z and w2 = u' y) on the block's pixels inside
// the image, to the work planes; u and y: the exposure's planes
template <int RY, int RX, bool STUDENT>
__device__ __forceinline__ void store_w(const Geom& g, const float (&acc)[RY][RX], int i0, int j0,
                                        const float* u, const float* y, float nu, float* w,
                                        float* w2) {
  const bool whole = j0 + RX <= g.W;
#pragma unroll
  for (int p = 0; p < RY; ++p) {
    if (i0 + p >= g.H) break;
    // B, P and the block's first column are even: pairs are 8-byte aligned
    const long long off = (long long)(g.B + i0 + p) * g.P + g.B + j0;
#pragma unroll
    for (int c = 0; c < RX; c += 2) {
      const float2 uu = __ldg(reinterpret_cast<const float2*>(u + off + c));
      float2 wv, w2v;
      if (STUDENT) {
        const float2 yy = __ldg(reinterpret_cast<const float2*>(y + off + c));
        const float s0 = student_weight(uu.x, yy.x, acc[p][c], nu);
        const float s1 = student_weight(uu.y, yy.y, acc[p][c + 1], nu);
        wv = make_float2(s0 * acc[p][c], s1 * acc[p][c + 1]);
        w2v = make_float2(s0 * yy.x, s1 * yy.y);
      } else {
        wv = make_float2(uu.x * acc[p][c], uu.y * acc[p][c + 1]);
      }
      if (whole) {
        *reinterpret_cast<float2*>(w + off + c) = wv;
        if (STUDENT) *reinterpret_cast<float2*>(w2 + off + c) = w2v;
      } else {
        if (j0 + c < g.W) w[off + c] = wv.x;
        if (j0 + c + 1 < g.W) w[off + c + 1] = wv.y;
        if (STUDENT) {
          if (j0 + c < g.W) w2[off + c] = w2v.x;
          if (j0 + c + 1 < g.W) w2[off + c + 1] = w2v.y;
        }
      }
    }
  }
}

// one pixel of Eq. (2) (the expressions of halo_kernel)
__device__ __forceinline__ float em_update(float xo, float d, float n) {
  float xv = xo;
  if (d > 0.f) {
    const float nv = fmaxf(n, 0.f);
    if (d < 1e-30f)  // denominator near zero: guarded ratio in FP64
      xv = (float)((double)xo * (double)nv / (double)d);
    else
      xv = xo * nv / d;
  }
  return xv;
}

// Adds the partial planes part[pass][e] (e < ne) of one phase into Den (and
// N') in exposure order on the block's pixels, and stores them or, after the
// last exposures, applies the update. first: the exposures before were none.
//
// Every load of a block of rows comes before its first store (x' may alias
// what is read, so the compiler keeps their order): the sums of a block wait
// for memory once per exposure, not once per four pixels (128 x 128 x 4,
// K = 15: 32.2 -> 29.2 us an iteration).
template <int RY, int RX, bool STUDENT>
__device__ __forceinline__ void sum_parts(const Shape& s, const FusedArgs& a, const float* part,
                                          int ne, int phi, int i0, int j0, bool first, bool last) {
  constexpr int NP = STUDENT ? 2 : 1, NR = RX >= 16 ? 1 : RY;  // rows of a block
  const Geom& g = s.g;
  const long long pb = (long long)phi * g.plane, step = (long long)s.R2 * g.plane;
  // rows and columns past the image stay inside the padded planes
#pragma unroll 1
  for (int p0 = 0; p0 < RY; p0 += NR) {
    if (i0 + p0 >= g.H || j0 >= g.W) break;
    const long long off = pb + (long long)(g.B + i0 + p0) * g.P + g.B + j0;
    float d[NP][NR][RX], xo[NR][RX], nn[NR][RX];
#pragma unroll
    for (int p = 0; p < NR; ++p)
#pragma unroll
      for (int c = 0; c < RX; ++c) {
        const long long o = off + (long long)p * g.P + c;
        xo[p][c] = last ? __ldcg(a.x + o) : 0.f;
        nn[p][c] = last && !STUDENT ? a.N[o] : 0.f;
#pragma unroll
        for (int q = 0; q < NP; ++q)
          d[q][p][c] = first ? 0.f : __ldcg((q == 0 ? a.Den : a.Nw) + o);
      }
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const float* src = part + (long long)q * ne * step + off;
#pragma unroll 2
      for (int e = 0; e < ne; ++e)
#pragma unroll
        for (int p = 0; p < NR; ++p)
#pragma unroll
          for (int c = 0; c < RX; c += 2) {
            const float2 v =
                __ldcg(reinterpret_cast<const float2*>(src + e * step + (long long)p * g.P + c));
            d[q][p][c] = first && e == 0 ? v.x : d[q][p][c] + v.x;
            d[q][p][c + 1] = first && e == 0 ? v.y : d[q][p][c + 1] + v.y;
          }
    }
#pragma unroll
    for (int p = 0; p < NR; ++p) {
      if (i0 + p0 + p >= g.H) break;
#pragma unroll
      for (int c = 0; c < RX; ++c) {
        if (j0 + c >= g.W) break;
        const long long o = off + (long long)p * g.P + c;
        if (last) {
          const float n = STUDENT ? d[NP - 1][p][c] : nn[p][c];
          a.xn[o] = em_update(xo[p][c], d[0][p][c], n);
        } else {
#pragma unroll
          for (int q = 0; q < NP; ++q)
            (q == 0 ? a.Den : a.Nw)[o] = d[q][p][c];
        }
      }
    }
  }
}

template <int RY, int RX>
__device__ __forceinline__ void zero_block(float (&acc)[RY][RX]) {
#pragma unroll
  for (int p = 0; p < RY; ++p)
#pragma unroll
    for (int c = 0; c < RX; ++c) acc[p][c] = 0.f;
}

// stores the block's pixels inside the image into one plane
template <int RY, int RX>
__device__ __forceinline__ void store_block(const Geom& g, const float (&acc)[RY][RX], int i0,
                                            int j0, float* plane) {
  const bool whole = j0 + RX <= g.W;
#pragma unroll
  for (int p = 0; p < RY; ++p) {
    if (i0 + p >= g.H) break;
    float* dst = plane + (long long)(g.B + i0 + p) * g.P + g.B + j0;
#pragma unroll
    for (int c = 0; c < RX; c += 2) {
      if (whole) {
        *reinterpret_cast<float2*>(dst + c) = make_float2(acc[p][c], acc[p][c + 1]);
      } else {
        if (j0 + c < g.W) dst[c] = acc[p][c];
        if (j0 + c + 1 < g.W) dst[c + 1] = acc[p][c + 1];
      }
    }
  }
}

// The last CTA to bring its partial of a tile and phase (count of ne) returns
// true, with every partial visible to it; the counter is back at zero.
__device__ __forceinline__ bool last_to_arrive(int* counter, int ne, int* flag_s) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool last = atomicAdd(counter, 1) == ne - 1;
    if (last) *counter = 0;
    *flag_s = last;
  }
  __syncthreads();
  if (*flag_s) __threadfence();
  return *flag_s != 0;
}

// ---------------------------------------------------------------------------
// taps form
// ---------------------------------------------------------------------------

// Tile variants, 4 x 16 outputs per thread: 64 x 128 (128 threads) where the
// chunk fills the SMs several times over, 64 x 64 (64 threads) otherwise, whose
// items divide the SMs more evenly.
template <int V> struct TapsTile;
template <> struct TapsTile<0> { static constexpr int TH = 64, TW = 128, MINB = 3; };
template <> struct TapsTile<1> { static constexpr int TH = 64, TW = 64, MINB = 5; };

template <int V, class Taps>
constexpr int taps_min_blocks() {
  // taps in shared memory: halo_kernel's registers
  return std::is_same<Taps, TapBank>::value ? TapsTile<V>::MINB : V == 0 ? 2 : 4;
}

// floats of a staged window
__host__ __device__ inline int taps_window_floats(const Shape& s, int TH, int TW) {
  const int rows = TH + 2 * s.hc;
  return rows * (TW + s.KP) + 4 * ((rows + 3) / 4);
}

struct TapsArgs {
  FusedArgs a;      // t0, t1: all exposures of the iteration
  float* w;         // chunk planes (heavy-tailed: then chunk planes of w2)
  float* part;      // parts: chunk x R2 planes (heavy-tailed: twice)
  int c0, ne;       // exposures [c0, c0 + ne) of this launch
  int epi;          // exposures per forward item
  int parts;        // adjoint partials per exposure, summed by taps_sum_kernel
  int gx, T;        // tiles per row, tiles
};

template <int V, bool STUDENT, class Taps>
__global__ void __launch_bounds__(TapsTile<V>::TH / 4 * (TapsTile<V>::TW / 16),
                                  taps_min_blocks<V, Taps>())
    taps_forward_kernel(const Shape s, const TapsArgs A, const __grid_constant__ Taps bank) {
  constexpr int TH = TapsTile<V>::TH, TW = TapsTile<V>::TW, NY = TH / 4, NT = NY * (TW / 16);
  extern __shared__ __align__(128) float smem[];
  const Geom& g = s.g;
  const SPlane sp{smem, TW + s.KP};
  float* ks = smem + taps_window_floats(s, TH, TW);  // TapMemory
  const int my = threadIdx.x % NY, mx = threadIdx.x / NY;
  const int grp = blockIdx.x / A.T, k = blockIdx.x - grp * A.T;
  const int i0 = (k / A.gx) * TH, j0 = (k % A.gx) * TW;
  const int e1 = min(A.ne, (grp + 1) * A.epi);
  for (int e = grp * A.epi; e < e1; ++e) {
    float acc[4][16];
    zero_block(acc);
    for (int phi = 0; phi < s.R2; ++phi) {
      if (s.R2 > 1 || e == grp * A.epi) {
        __syncthreads();  // readers of the previous window are done
        stage_window<4, NT, 4, false>(
            sp, A.a.x + (long long)phi * g.plane + (long long)(i0 + s.hc) * g.P, g.P, j0 + s.hc,
            TH + 2 * s.hc, TW + s.KP);
        __syncthreads();
      }
      corr_launch<NT>(acc, sp, 4 * my, 16 * mx, bank, (e * s.R2 + phi) * s.Kc * s.KP, s.KP, s.Kc,
                      ks);
    }
    const long long tp = (long long)(A.c0 + e) * g.plane;
    store_w<4, 16, STUDENT>(g, acc, i0 + 4 * my, j0 + 16 * mx, A.a.u + tp, A.a.y + tp, A.a.nu,
                            A.w + (long long)e * g.plane, A.w + (long long)(A.ne + e) * g.plane);
  }
}

// blockIdx.x: tile, y: phase; z: exposure of the chunk (parts) or one CTA
// running all of them in order, adding each to Den (and N') in global memory
template <int V, bool STUDENT, class Taps>
__global__ void __launch_bounds__(TapsTile<V>::TH / 4 * (TapsTile<V>::TW / 16),
                                  taps_min_blocks<V, Taps>())
    taps_adjoint_kernel(const Shape s, const TapsArgs A, const __grid_constant__ Taps bank) {
  constexpr int TH = TapsTile<V>::TH, TW = TapsTile<V>::TW, NY = TH / 4, NT = NY * (TW / 16);
  extern __shared__ __align__(128) float smem[];
  const Geom& g = s.g;
  const SPlane sp{smem, TW + s.KP};
  float* ks = smem + taps_window_floats(s, TH, TW);  // TapMemory
  const int my = threadIdx.x % NY, mx = threadIdx.x / NY;
  const int k = blockIdx.x, phi = blockIdx.y;
  const int i0 = (k / A.gx) * TH, j0 = (k % A.gx) * TW;
  const int i = i0 + 4 * my, j = j0 + 16 * mx;
  const long long pb = (long long)phi * g.plane;
  const bool first = A.c0 == A.a.t0, last = A.c0 + A.ne == A.a.t1;
  const int e0 = A.parts ? blockIdx.z : 0, e1 = A.parts ? e0 + 1 : A.ne;
  for (int e = e0; e < e1; ++e) {
#pragma unroll 1
    for (int pass = 0; pass < (STUDENT ? 2 : 1); ++pass) {
      float acc[4][16];
      zero_block(acc);
      __syncthreads();  // readers of the previous window are done
      stage_window<4, NT, 4, false>(
          sp, A.w + (long long)(pass * A.ne + e) * g.plane + (long long)(i0 + s.hc) * g.P, g.P,
          j0 + s.hc, TH + 2 * s.hc, TW + s.KP);
      __syncthreads();
      corr_launch<NT>(acc, sp, 4 * my, 16 * mx, bank, (e * s.R2 + phi) * s.Kc * s.KP, s.KP, s.Kc,
                      ks);
      if (A.parts) {
        store_block(g, acc, i, j, A.part + (long long)(pass * A.ne + e) * s.R2 * g.plane + pb);
        continue;
      }
      float* run = (pass == 0 ? A.a.Den : A.a.Nw) + pb;
      const bool begin = first && e == 0, end = last && e + 1 == A.ne;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if (i + p >= g.H) break;
        const long long off = (long long)(g.B + i + p) * g.P + g.B + j;
        // columns past the image stay inside the padded plane
        float2* run2 = reinterpret_cast<float2*>(run + off);
        if (!begin) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const float2 v = run2[c];
            acc[p][2 * c] = v.x + acc[p][2 * c];
            acc[p][2 * c + 1] = v.y + acc[p][2 * c + 1];
          }
        }
        // not the last exposure; or the heavy-tailed Den, kept for pass 1
        // (read back below by the thread that wrote it)
        if (!end || (STUDENT && pass == 0)) {
#pragma unroll
          for (int c = 0; c < 8; ++c) run2[c] = make_float2(acc[p][2 * c], acc[p][2 * c + 1]);
          continue;
        }
#pragma unroll
        for (int c = 0; c < 16; ++c)
          if (j + c < g.W) {
            const float d = STUDENT ? A.a.Den[pb + off + c] : acc[p][c];
            const float n = STUDENT ? acc[p][c] : A.a.N[pb + off + c];
            A.a.xn[pb + off + c] = em_update(A.a.x[pb + off + c], d, n);
          }
      }
    }
  }
}

// parts: adds the chunk's partials in exposure order, one row of 4 x 128 pixels
// per CTA (blockIdx.y: row, z: phase). A launch of its own: counting the items
// of a tile in instead costs every item a fence and an atomic round trip.
template <bool STUDENT>
__global__ void __launch_bounds__(128) taps_sum_kernel(const Shape s, const TapsArgs A) {
  const int j = 4 * (blockIdx.x * 128 + threadIdx.x);
  if (j < s.g.W)
    sum_parts<1, 4, STUDENT>(s, A.a, A.part, A.ne, blockIdx.z, blockIdx.y, j, A.c0 == A.a.t0,
                             A.c0 + A.ne == A.a.t1);
}

// ---------------------------------------------------------------------------
// split form
// ---------------------------------------------------------------------------

// Tile variants: 2 x RX outputs per thread. Fewer outputs per thread cost more
// shared loads per FMA and more staging per output, but give more warps.
template <int V> struct SplitTile;
template <> struct SplitTile<0> { static constexpr int TH = 32, TW = 64, RX = 16; };
template <> struct SplitTile<1> { static constexpr int TH = 32, TW = 32, RX = 8; };

struct SplitArgs {
  FusedArgs a;      // x, xn: current and next buffers of the first iteration
  float* w;         // chunk planes (heavy-tailed: then chunk planes of w2)
  float* part;      // chunk x R2 planes (heavy-tailed: twice)
  int* ctrl;        // [0] barrier arrivals, [1] CTAs finished, [2] abort flag
  int* counters;    // one per (phase, tile)
  int chunk, iters;
  int gx, T;
};

template <int V, bool STUDENT>
__global__ void __launch_bounds__(SplitTile<V>::TH / 2 * (SplitTile<V>::TW / SplitTile<V>::RX))
    split_kernel(const Shape s, const SplitArgs A) {
  constexpr int TH = SplitTile<V>::TH, TW = SplitTile<V>::TW, RX = SplitTile<V>::RX;
  constexpr int NY = TH / 2, NT = NY * (TW / RX);
  extern __shared__ __align__(128) float smem[];
  __shared__ int flag_s;
  const Geom& g = s.g;
  const int rows = TH + 2 * s.hc, cols = TW + s.KP, kf4 = s.Kc * s.KP >> 2;
  const SPlane sp{smem, cols};
  float* ks = smem + rows * cols + 4 * ((rows + 1) >> 1);
  const int my = threadIdx.x % NY, mx = threadIdx.x / NY;
  const int n = A.a.t1 - A.a.t0;
  FusedArgs a = A.a;
  int round = 0;
  bool ok = true;
  auto stage = [&](const float* plane, const float* taps, int i0, int j0) {
    __syncthreads();  // readers of the previous window and taps are done
    stage_window<2, NT, 4, true>(sp, plane + (long long)(i0 + s.hc) * g.P, g.P, j0 + s.hc, rows,
                                 cols);
    const float4* kg = reinterpret_cast<const float4*>(taps);
    for (int q = threadIdx.x; q < kf4; q += NT) reinterpret_cast<float4*>(ks)[q] = __ldg(kg + q);
    __syncthreads();
  };
  for (int it = 0; ok && it < A.iters; ++it) {
    for (int c0 = 0; ok && c0 < n; c0 += A.chunk) {
      const int ne = min(A.chunk, n - c0);
      const bool first = c0 == 0, last = c0 + ne == n;
      for (int id = blockIdx.x; id < ne * A.T; id += gridDim.x) {
        const int e = id / A.T, k = id - e * A.T, t = a.t0 + c0 + e;
        const int i0 = (k / A.gx) * TH, j0 = (k % A.gx) * TW;
        float acc[2][RX];
        zero_block(acc);
        for (int phi = 0; phi < s.R2; ++phi) {
          stage(a.x + (long long)phi * g.plane,
                a.kf + ((long long)t * s.R2 + phi) * s.Kc * s.KP, i0, j0);
          corr_tile<2, RX>(acc, sp, 2 * my, RX * mx, ks, s.KP, s.Kc);
        }
        const long long tp = (long long)t * g.plane;
        store_w<2, RX, STUDENT>(g, acc, i0 + 2 * my, j0 + RX * mx, a.u + tp, a.y + tp, a.nu,
                                A.w + (long long)e * g.plane,
                                A.w + (long long)(ne + e) * g.plane);
      }
      ok = grid_barrier(A.ctrl, ++round, &flag_s);
      const int per = A.T * s.R2;
      for (int id = blockIdx.x; ok && id < ne * per; id += gridDim.x) {
        const int e = id / per, rest = id - e * per, phi = rest / A.T, k = rest - phi * A.T;
        const int t = a.t0 + c0 + e;
        const int i0 = (k / A.gx) * TH, j0 = (k % A.gx) * TW;
#pragma unroll 1
        for (int pass = 0; pass < (STUDENT ? 2 : 1); ++pass) {
          float acc[2][RX];
          zero_block(acc);
          stage(A.w + (long long)(pass * ne + e) * g.plane,
                a.ka + ((long long)t * s.R2 + phi) * s.Kc * s.KP, i0, j0);
          corr_tile<2, RX>(acc, sp, 2 * my, RX * mx, ks, s.KP, s.Kc);
          store_block(g, acc, i0 + 2 * my, j0 + RX * mx,
                      A.part + (long long)((pass * ne + e) * s.R2 + phi) * g.plane);
        }
        if (last_to_arrive(A.counters + rest, ne, &flag_s))
          sum_parts<2, RX, STUDENT>(s, a, A.part, ne, phi, i0 + 2 * my, j0 + RX * mx, first, last);
      }
      if (ok) ok = grid_barrier(A.ctrl, ++round, &flag_s);
    }
    float* t = const_cast<float*>(a.x);
    a.x = a.xn;
    a.xn = t;
  }
  // the last CTA leaves the control words (and, after a wait that gave up, the
  // tile counters) at zero for the next launch
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!ok) atomicOr(a.err, kErrTimeout);
    __threadfence();
    flag_s = atomicAdd(&A.ctrl[1], 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (flag_s) {
    __threadfence();
    if (!ok)
      for (int q = threadIdx.x; q < A.T * s.R2; q += NT) A.counters[q] = 0;
    if (threadIdx.x < 3) A.ctrl[threadIdx.x] = 0;
  }
}

size_t taps_smem_bytes(const Shape& s, int TH, int TW) {
  return (size_t)taps_window_floats(s, TH, TW) * sizeof(float);
}

size_t split_smem_bytes(const Shape& s, int TH, int TW) {
  const int rows = TH + 2 * s.hc;
  return ((size_t)rows * (TW + s.KP) + 4 * ((rows + 1) / 2) + (size_t)s.Kc * s.KP) * sizeof(float);
}

int cdiv(int a, int b) { return (a + b - 1) / b; }

// ---------------------------------------------------------------------------
// the numerator N = sum_t F_t^T (u_t y_t)
// ---------------------------------------------------------------------------

// One adjoint pass in the taps form, its windows staged as products u y straight
// from the planes (no work planes). It runs once per frame set, and its rounding
// stays in every iterate: the taps are summed in blocks (corr_tile). Images whose
// tiles do not fill the SMs run up to kNumParts + 1 exposures side by side: the
// first adds to N in place, the others' sums go to planes that are scratch at that
// time, and a second launch adds those in exposure order (33 x 1024^2, K = 43, set-up
// and log-likelihood included: 6.73 ms with three such planes, 6.89 with one).
struct NumeratorArgs {
  const float *u, *y;     // n planes
  float* N;               // R2 planes
  float* part[kNumParts]; // R2 planes each
  int c0, ne;             // exposures [c0, c0 + ne) of this launch
  int parts;              // one exposure per blockIdx.z: 0 into N, z into part[z - 1]
  int gx;                 // tiles per row
};

// CTAS per SM: the block sums need 240 registers, or 168 and a few spills, which
// more CTAs on an SM outweigh (21 x 814 x 895, K = 15: 826 -> 720 us a frame set;
// 24 x 900^2, K = 29: 1592 -> 1316; 4096^2 x 9, K = 43: 12.60 -> 12.31 ms) except on
// 64 x 64 tiles whose windows leave shared memory for four only (33 x 1024^2, K = 43:
// 5 % slower with 168).
template <int V, int CTAS>
__global__ void __launch_bounds__(TapsTile<V>::TH / 4 * (TapsTile<V>::TW / 16), CTAS)
    taps_numerator_kernel(const Shape s, const __grid_constant__ NumeratorArgs A,
                          const __grid_constant__ TapBank bank) {
  constexpr int TH = TapsTile<V>::TH, TW = TapsTile<V>::TW, NY = TH / 4, NT = NY * (TW / 16);
  extern __shared__ __align__(128) float smem[];
  const Geom& g = s.g;
  const SPlane sp{smem, TW + s.KP};
  const int my = threadIdx.x % NY, mx = threadIdx.x / NY;
  const int k = blockIdx.x, phi = blockIdx.y;
  const int i0 = (k / A.gx) * TH, j0 = (k % A.gx) * TW;
  const int i = i0 + 4 * my, j = j0 + 16 * mx;
  const long long pb = (long long)phi * g.plane;
  const int e0 = A.parts ? blockIdx.z : 0, e1 = A.parts ? e0 + 1 : A.ne;
  for (int e = e0; e < e1; ++e) {
    const long long row0 = (long long)(A.c0 + e) * g.plane + (long long)(i0 + s.hc) * g.P;
    const float *u = A.u + row0, *y = A.y + row0;
    __syncthreads();  // readers of the previous window are done
    stage_words<4, NT, 4>(
        sp,
        [u, y](long long off) {
          const float4 a = __ldg(reinterpret_cast<const float4*>(u + off));
          const float4 b = __ldg(reinterpret_cast<const float4*>(y + off));
          return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
        },
        g.P, j0 + s.hc, TH + 2 * s.hc, TW + s.KP);
    __syncthreads();
    float acc[4][16];
    zero_block(acc);
    corr_bank<true>(acc, sp, 4 * my, 16 * mx, bank, (e * s.R2 + phi) * s.Kc * s.KP, s.KP, s.Kc);
    const bool in_place = !A.parts || e == 0;
    if (in_place && A.c0 + e > 0) {
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int c = 0; c < 16; ++c)
          if (i + p < g.H && j + c < g.W)
            acc[p][c] += A.N[pb + (long long)(g.B + i + p) * g.P + g.B + j + c];
    }
    store_block(g, acc, i, j, (in_place ? A.N : A.part[e - 1]) + pb);
  }
}

// N += the launch's parts in exposure order, rows of pixels by pairs
__global__ void __launch_bounds__(128)
    numerator_sum_kernel(const Shape s, const NumeratorArgs A) {
  const int j = 2 * (blockIdx.x * 128 + threadIdx.x);
  if (j >= s.g.W) return;
  const long long off =
      blockIdx.z * s.g.plane + (long long)(s.g.B + blockIdx.y) * s.g.P + s.g.B + j;
  float2 v = *reinterpret_cast<const float2*>(A.N + off);
#pragma unroll
  for (int e = 0; e < kNumParts; ++e)
    if (e + 1 < A.ne) {
      const float2 t = *reinterpret_cast<const float2*>(A.part[e] + off);
      v.x += t.x;
      v.y += t.y;
    }
  A.N[off] = v.x;
  if (j + 1 < s.g.W) A.N[off + 1] = v.y;
}

template <int V, int CTAS>
cudaError_t launch_numerator_t(const Shape& s, NumeratorArgs A, int chunk, const float* hka,
                               cudaStream_t st) {
  constexpr int TH = TapsTile<V>::TH, TW = TapsTile<V>::TW, NT = TH / 4 * (TW / 16);
  cudaError_t e = allow_max_dynamic_smem((const void*)taps_numerator_kernel<V, CTAS>);
  if (e != cudaSuccess) return e;
  const size_t smem = taps_smem_bytes(s, TH, TW), kfl = (size_t)s.R2 * s.Kc * s.KP;
  A.gx = cdiv(s.W, TW);
  const int T = A.gx * cdiv(s.H, TH);
  TapBank bank;
  for (A.c0 = 0; A.c0 < s.n; A.c0 += chunk) {
    A.ne = std::min(chunk, s.n - A.c0);
    std::copy(hka + (size_t)A.c0 * kfl, hka + (size_t)(A.c0 + A.ne) * kfl, bank.k);
    taps_numerator_kernel<V, CTAS><<<dim3(T, s.R2, A.parts ? A.ne : 1), NT, smem, st>>>(s, A, bank);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (A.parts && A.ne > 1) {
      numerator_sum_kernel<<<dim3(cdiv(s.W, 256), s.H, s.R2), 128, 0, st>>>(s, A);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// The log-likelihood's data term over the chunk (Eq. (1); the Student-t term
// with STUDENT): part[group * T + tile] (+)= sum of u (y - z)^2 in FP64 over
// the group's exposures, z as the forward pass computes it. Launches of later
// chunks add to the same partial sums, so their order is fixed.
template <int V, bool STUDENT>
__global__ void __launch_bounds__(TapsTile<V>::TH / 4 * (TapsTile<V>::TW / 16), TapsTile<V>::MINB)
    taps_chi2_kernel(const Shape s, const TapsArgs A, double* __restrict__ part,
                     const __grid_constant__ TapBank bank) {
  constexpr int TH = TapsTile<V>::TH, TW = TapsTile<V>::TW, NY = TH / 4, NT = NY * (TW / 16);
  extern __shared__ __align__(128) float smem[];
  __shared__ double red[NT / 32];
  const Geom& g = s.g;
  const SPlane sp{smem, TW + s.KP};
  const int my = threadIdx.x % NY, mx = threadIdx.x / NY;
  const int grp = blockIdx.x / A.T, k = blockIdx.x - grp * A.T;
  const int i0 = (k / A.gx) * TH, j0 = (k % A.gx) * TW;
  const int i = i0 + 4 * my, j = j0 + 16 * mx;
  const int e1 = min(A.ne, (grp + 1) * A.epi);
  double chi = 0.0;
  for (int e = grp * A.epi; e < e1; ++e) {
    float acc[4][16];
    zero_block(acc);
    for (int phi = 0; phi < s.R2; ++phi) {
      if (s.R2 > 1 || e == grp * A.epi) {
        __syncthreads();  // readers of the previous window are done
        stage_window<4, NT, 4, false>(
            sp, A.a.x + (long long)phi * g.plane + (long long)(i0 + s.hc) * g.P, g.P, j0 + s.hc,
            TH + 2 * s.hc, TW + s.KP);
        __syncthreads();
      }
      corr_bank(acc, sp, 4 * my, 16 * mx, bank, (e * s.R2 + phi) * s.Kc * s.KP, s.KP, s.Kc);
    }
    const long long tp = (long long)(A.c0 + e) * g.plane;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      if (i + p >= g.H) break;
      const long long off = tp + (long long)(g.B + i + p) * g.P + g.B + j;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const float uv = A.a.u[off + c];
        if (j + c < g.W && uv != 0.f) {
          const double d = (double)A.a.y[off + c] - (double)acc[p][c];
          if (STUDENT)
            chi += ((double)A.a.nu + 1.0) * log1p((double)uv * d * d / (double)A.a.nu);
          else
            chi += (double)uv * d * d;
        }
      }
    }
  }
  const double tot = block_sum_f64(chi, red);
  if (threadIdx.x == 0) part[blockIdx.x] = (A.c0 == A.a.t0 ? 0.0 : part[blockIdx.x]) + tot;
}

template <int V, bool STUDENT>
cudaError_t launch_chi2_t(const Shape& s, const FusedArgs& a, const float* hkf,
                          double* part, int max_parts, int* nparts, cudaStream_t st) {
  constexpr int TH = TapsTile<V>::TH, TW = TapsTile<V>::TW, NT = TH / 4 * (TW / 16);
  const size_t smem = taps_smem_bytes(s, TH, TW);
  cudaError_t e = allow_max_dynamic_smem((const void*)taps_chi2_kernel<V, STUDENT>);
  if (e != cudaSuccess) return e;
  const size_t kfl = (size_t)s.R2 * s.Kc * s.KP;
  TapsArgs A{};
  A.a = a;
  A.gx = cdiv(s.W, TW);
  A.T = A.gx * cdiv(s.H, TH);
  const int chunk = std::min(s.n, tap_bank_kernels(s) / s.R2);
  const int groups = std::min(chunk, max_parts / A.T);
  if (groups < 1) return cudaErrorInvalidValue;
  A.epi = cdiv(chunk, groups);
  *nparts = cdiv(chunk, A.epi) * A.T;
  TapBank bank;
  for (A.c0 = a.t0; A.c0 < a.t1; A.c0 += chunk) {
    A.ne = std::min(chunk, a.t1 - A.c0);
    std::copy(hkf + (size_t)A.c0 * kfl, hkf + (size_t)(A.c0 + A.ne) * kfl, bank.k);
    taps_chi2_kernel<V, STUDENT><<<A.T * cdiv(A.ne, A.epi), NT, smem, st>>>(s, A, part, bank);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void set_taps(TapBank& bank, const float* host, const float*, size_t first, size_t count) {
  std::copy(host + first, host + first + count, bank.k);
}
void set_taps(TapMemory& mem, const float*, const float* dev, size_t first, size_t) {
  mem.k = dev + first;
}

template <int V, bool STUDENT, class Taps>
cudaError_t launch_taps_t(const Shape& s, const DirectPlan& p, const DirectLaunch& h,
                          const float* hkf, const float* hka, cudaStream_t st) {
  constexpr int TH = TapsTile<V>::TH, TW = TapsTile<V>::TW, NT = TH / 4 * (TW / 16);
  const size_t smem = taps_smem_bytes(s, TH, TW) +
                      (std::is_same<Taps, TapBank>::value ? 0 : s.Kc * s.KP * sizeof(float));
  const auto forward = taps_forward_kernel<V, STUDENT, Taps>;
  const auto adjoint = taps_adjoint_kernel<V, STUDENT, Taps>;
  cudaError_t e = allow_max_dynamic_smem((const void*)forward);
  if (e == cudaSuccess) e = allow_max_dynamic_smem((const void*)adjoint);
  if (e != cudaSuccess) return e;
  const size_t kfl = (size_t)s.R2 * s.Kc * s.KP;  // taps of one exposure
  TapsArgs A;
  A.a = h.a;
  A.w = h.work;
  A.parts = p.parts;
  A.gx = cdiv(s.W, TW);
  A.T = A.gx * cdiv(s.H, TH);
  Taps bank;
  for (int c0 = h.a.t0; c0 < h.a.t1; c0 += p.chunk) {
    A.c0 = c0;
    A.ne = std::min(p.chunk, h.a.t1 - c0);
    A.part = h.work + (long long)(STUDENT ? 2 : 1) * A.ne * s.g.plane;
    // exposures per forward item (r = 1: its window is staged once): as many
    // as still leave 16 items an SM
    A.epi = s.R2 > 1 ? 1 : std::max(1, std::min(A.ne, A.T * A.ne / (16 * kSMs)));
    set_taps(bank, hkf, h.a.kf, c0 * kfl, A.ne * kfl);
    forward<<<A.T * cdiv(A.ne, A.epi), NT, smem, st>>>(s, A, bank);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    set_taps(bank, hka, h.a.ka, c0 * kfl, A.ne * kfl);
    adjoint<<<dim3(A.T, s.R2, p.parts ? A.ne : 1), NT, smem, st>>>(s, A, bank);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (p.parts) {
      taps_sum_kernel<STUDENT><<<dim3(cdiv(s.W, 512), s.H, s.R2), 128, 0, st>>>(s, A);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

template <class Taps>
cudaError_t launch_taps_of(const Shape& s, const DirectPlan& p, const DirectLaunch& h,
                           const float* hkf, const float* hka, cudaStream_t st) {
  if (h.a.nu > 0.f)
    return p.tile == 0 ? launch_taps_t<0, true, Taps>(s, p, h, hkf, hka, st)
                       : launch_taps_t<1, true, Taps>(s, p, h, hkf, hka, st);
  return p.tile == 0 ? launch_taps_t<0, false, Taps>(s, p, h, hkf, hka, st)
                     : launch_taps_t<1, false, Taps>(s, p, h, hkf, hka, st);
}

template <int V, bool STUDENT>
cudaError_t launch_split_t(const Shape& s, const DirectPlan& p, const DirectLaunch& h, float* xa,
                           float* xb, int iters, cudaStream_t st) {
  constexpr int NT = SplitTile<V>::TH / 2 * (SplitTile<V>::TW / SplitTile<V>::RX);
  const size_t smem = split_smem_bytes(s, SplitTile<V>::TH, SplitTile<V>::TW);
  const void* kern = (const void*)split_kernel<V, STUDENT>;
  cudaError_t e = allow_max_dynamic_smem(kern);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, occ = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, smem)) != cudaSuccess)
    return e;
  SplitArgs A;
  A.a = h.a;
  A.a.x = xa;
  A.a.xn = xb;
  A.chunk = p.chunk;
  A.iters = iters;
  A.w = h.work;
  A.part = h.work + (long long)(STUDENT ? 2 : 1) * p.chunk * s.g.plane;
  A.ctrl = h.counters;
  A.counters = h.counters + 64;
  A.gx = cdiv(s.W, SplitTile<V>::TW);
  A.T = A.gx * cdiv(s.H, SplitTile<V>::TH);
  const long long items = (long long)std::min(p.chunk, h.a.t1 - h.a.t0) * A.T * s.R2;
  const int grid = (int)std::min<long long>(items, (long long)sms * std::max(occ, 1));
  void* args[2] = {const_cast<Shape*>(&s), &A};
  return cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(NT), args, smem, st);
}

}  // namespace

int tap_bank_kernels(const Shape& s) { return kTapFloats / (s.Kc * s.KP); }

int direct_counter_ints(const Shape& s) {
  return 64 + s.R2 * cdiv(s.W, 32) * cdiv(s.H, 32);  // of the smaller tiles
}

cudaError_t launch_taps_iter(const Shape& s, const DirectPlan& p, const DirectLaunch& h,
                             const float* hkf, const float* hka, cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const cudaError_t e = cudaStreamIsCapturing(st, &cap);
  if (e != cudaSuccess) return e;
  return cap == cudaStreamCaptureStatusNone ? launch_taps_of<TapBank>(s, p, h, hkf, hka, st)
                                            : launch_taps_of<TapMemory>(s, p, h, hkf, hka, st);
}

int numerator_exposures(const Shape& s) {
  return s.Kc >= 5 ? std::min(s.n, tap_bank_kernels(s) / s.R2) : 0;
}

cudaError_t launch_numerator(const Shape& s, const float* u, const float* y, const float* hka,
                             float* N, float* const (&part)[kNumParts], cudaStream_t st) {
  NumeratorArgs A{};
  A.u = u;
  A.y = y;
  A.N = N;
  std::copy(part, part + kNumParts, A.part);
  // the rules of direct_plan: parts where tiles and phases alone do not fill the SMs,
  // 64 x 64 tiles for few items
  const long long T = (long long)s.gx * cdiv(s.H, 64);
  A.parts = T * s.R2 < 4 * kSMs;
  const int most = numerator_exposures(s), chunk = A.parts ? std::min(most, kNumParts + 1) : most;
  if (T * chunk >= 1500) return launch_numerator_t<0, 3>(s, A, chunk, hka, st);
  return 6 * (taps_smem_bytes(s, 64, 64) + 1024) <= 228 * 1024
             ? launch_numerator_t<1, 6>(s, A, chunk, hka, st)
             : launch_numerator_t<1, 4>(s, A, chunk, hka, st);
}

cudaError_t launch_taps_chi2(const Shape& s, const DirectPlan& p, const FusedArgs& a,
                             const float* hkf, double* part, int max_parts, int* nparts,
                             cudaStream_t st) {
  if (a.nu > 0.f)
    return p.tile == 0 ? launch_chi2_t<0, true>(s, a, hkf, part, max_parts, nparts, st)
                       : launch_chi2_t<1, true>(s, a, hkf, part, max_parts, nparts, st);
  return p.tile == 0 ? launch_chi2_t<0, false>(s, a, hkf, part, max_parts, nparts, st)
                     : launch_chi2_t<1, false>(s, a, hkf, part, max_parts, nparts, st);
}

cudaError_t launch_split_iters(const Shape& s, const DirectPlan& p, const DirectLaunch& h,
                               float* xa, float* xb, int iters, cudaStream_t st) {
  if (h.a.nu > 0.f)
    return p.tile == 0 ? launch_split_t<0, true>(s, p, h, xa, xb, iters, st)
                       : launch_split_t<1, true>(s, p, h, xa, xb, iters, st);
  return p.tile == 0 ? launch_split_t<0, false>(s, p, h, xa, xb, iters, st)
                     : launch_split_t<1, false>(s, p, h, xa, xb, iters, st);
}

int split_iters_per_launch(const Shape& s) {
  // about 2 ms a launch (20 TFLOP/s and 20 us of barriers an iteration), so
  // that other streams' work is not held up longer
  const double us = 20.0 + 6.0 * s.n * s.R2 * (double)s.H * s.W * s.Kc * s.Kc / 20e6;
  return std::max(1, (int)(2000.0 / us));
}

namespace {

// Work planes a context may take: half as many as it holds anyway, or 64 MB where
// that is more (small images, whose planes are small and whose items few).
long long plane_budget(const Shape& s) {
  const long long planes = 2LL * s.n + 4LL * s.R2;
  return std::max(planes / 2, (64LL << 20) / (s.g.plane * (long long)sizeof(float)));
}

// exposures per chunk of `per` planes each: `want`, or what the budget allows, in
// chunks of about equal size
int fit_chunk(const Shape& s, int want, int per) {
  const long long budget = plane_budget(s);
  if ((long long)want * per <= budget) return want;
  const int most = (int)std::max(1LL, budget / per);
  return cdiv(s.n, cdiv(s.n, most));
}

}  // namespace

DirectPlan direct_plan(const Shape& s, bool student) {
  DirectPlan p{};
  const long long T = (long long)s.gx * cdiv(s.H, 64);  // 64 x 128 tiles
  const int cap = s.Kc >= 5 ? tap_bank_kernels(s) / s.R2 : 0;  // exposures of one launch
  // one CTA per tile and phase adds the exposures itself where those fill
  // the SMs; else their partials take planes (2048^2 15, 8: 967 and 909 us;
  // 1600 x 1500: 3352 and 3358; 4096^2: 62670 and 66560)
  const int parts = T * s.R2 < 4 * kSMs;
  // Exposures of a taps launch: 8192 items (18 waves of three CTAs an SM)
  // leave little of a last wave idle; more would only take memory for w.
  int taps = (int)std::min<long long>({(long long)cap, (long long)s.n,
                                       std::max(4LL, 8192 / T)});
  taps = std::min(taps, fit_chunk(s, taps, 1 + parts * s.R2));
  // The split form's 32 x 64 tiles, or 32 x 32 tiles with half the outputs per thread
  // where even those give few warps (300^2 21, 12, 1.1 M outputs an operator: 106 and
  // 90 us; 512^2 31, 12, 3.2 M: 342 and 389)
  const int split_tile = (double)s.n * s.R2 * s.H * s.W >= 2e6 ? 0 : 1;
  const int split = fit_chunk(s, s.n, 1 + s.R2);
  const long long split_items = (long long)split * cdiv(s.W, split_tile == 0 ? 64 : 32) * cdiv(s.H, 32);
  // Measured (us an iteration, halo / taps / split; K, n): 128^2 15, 4: 166 /
  // 78 / 29; 300^2 21, 12: 735 / 156 / 90; 512^2 31, 12 (T taps = 280): 1201 /
  // 450 / 342; 700 x 800 31, 20 (539): 2035 / 1075 / 1101; 1021 x 1009 43, 33
  // (512): 6196 / 5675 / 5660; 1600 x 1500 31, 20: 4171 / 3352 / 4228; 4096^2
  // 43, 33: 80173 / 62670 / 93051. Below 500 items a taps launch leaves SMs
  // idle and the split form, with every exposure's items in one phase, wins; where
  // its planes are over the budget, while a chunk still has two items an SM. From 100
  // tiles on it loses to halo_kernel's 32-row tiles (us, split / halo; K, n, r: 900 x
  // 1000 43, 10: 2332 / 1581; 1100 x 1150 47, 20: 5962 / 4620; 1000^2 47, 31, 8: 40426
  // / 23371; 900^2 93, 12, 2: 10899 / 8411; 800^2, T = 91, 43, 24: 3378 / 3038; 700^2,
  // T = 66, 43, 24: 2336 / 2722), except with kernels below 5 x 5, whose windows cost
  // little (1200^2 3, 12: 263 / 278; 1900^2, T = 450, 3, 4: 246 / 223).
  if (taps > 0 && T * taps >= 500) {
    p.form = kFormTaps;
    p.chunk = taps;
    p.parts = parts;
    // 64 x 64 tiles divide few items more evenly (700 x 800: 1123 and 1075 us;
    // 1600 x 1500, 2100 items: 3352 and 3434)
    p.tile = T * taps >= 1500 ? 0 : 1;
  } else if (T * s.n < 4000 && T < (s.Kc >= 5 ? 100 : 500) && (split == s.n || split_items >= 2 * kSMs)) {
    p.form = kFormSplit;
    p.parts = 1;
    p.chunk = split;
    p.tile = split_tile;
  } else {
    return p;  // halo_kernel: no work planes
  }
  const int per = 1 + p.parts * s.R2;  // planes per exposure (heavy-tailed: twice as many)
  p.planes = std::max(p.chunk, 2) * per;
  if (student) p.chunk = std::min(p.chunk, p.planes / (2 * per));
  return p;
}

}  // namespace emd
