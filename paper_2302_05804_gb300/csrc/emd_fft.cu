// emd_fft.cu -- the forward model and the adjoint of Eq. (2) by FFT
// (overlap-save on 128 x 128 tiles), an alternative to the direct FP32
// kernels. Same arithmetic type (FP32), different rounding. For r > 1 every
// operator below acts on the polyphase planes with the Kc x Kc phase
// kernels (hc in place of h), summed over the phases in the forward model.
//
// For an output tile with origin (i0, j0) and side B = 128 - 2 hc (hc =
// (K-1)/2), the input region is rows/cols [i0 - hc, i0 - hc + 128) of the
// image, zero outside it. With k the K x K PSF at the top-left of a zero
// 128 x 128 array, the circular convolution of the region with k holds
// z(i0 + p, j0 + q) at circular index (p + 2hc, q + 2hc), and the circular
// correlation of the w region with k holds Den(i0 + p, j0 + q) at (p, q),
// for p, q < B: no wrapped term reaches those indices.
//
// Two exposures share one complex transform, without splitting or merging.
// With the complex kernel k = k_a + i k_b:
//   forward  IFFT(x^ k^) = z_a + i z_b;
//   adjoint  the real part of IFFT(FFT(w_a + i w_b) conj(k^)) is
//            corr(w_a, k_a) + corr(w_b, k_b), which is all Den needs (the
//            imaginary part holds cross terms and is dropped).
// The rounding of one exposure's half is of the size of the other's, so the two
// kernels are brought to the same size first: k_t stands for s_t k_t, s_t the power
// of two (exact) that takes the kernel's sum nearest to 1, and the forward pass
// divides it out again (PSFs may carry the exposures' flux scales). The spectra
// also carry the 1 / 128^2 of the inverse transforms.
// Heavy-tailed noise packs the two images of one exposure instead: with the
// real kernel k_t, IFFT(FFT(w + i w2) conj(k_t^)) = Den_t + i N'_t. There, too, one
// half's rounding is of the other's size, and far from convergence the data
// exceed the model by any factor: w2 is brought to w's size by a power of two per
// tile (student_scale), taken out of N' again.
// x is real, so x^(-m, -f) = conj(x^(m, f)): 64 column slots (m = 1 .. 63, and
// columns 0 and 64 in slot 0) stand for the 128 columns. Slot m serves the
// columns m and 128 - m, the second by conjugation:
//   forward  column 128 - m after the inverse transform over f is
//            conj(IFFT_f(x^(m, f) S2(m, f))), S2(m, f) = conj(k^(128-m, -f));
//   adjoint  the Hermitian part of the product, H(m, f) = Z(m, f) conj(S1(m, f))
//            + FFT_f(conj(column 128 - m)) conj(S2(m, f)), S1 = k^.
// So a slot's spectrum values, x^ or the accumulator H, are 16 complex
// registers per thread for all exposures, and the tables S1 and S2 are
// read once per pair.
//
// A 128-point FFT is eight lanes' work, 16 values each: a 16-point DFT in
// registers (inputs j + 8 i of lane j), twiddles, one exchange through the
// row's or column's own shared memory, two 8-point DFTs. Frequencies 2 t + 16 q
// and 2 t + 1 + 16 q end in lane t (adjacent: rows move them as 16-byte words);
// the inverse takes them there and runs the stages in reverse. The exchange
// positions, the row pitch of 130 complex and the choice of a warp's four rows
// and columns (Lane) keep every access free of bank conflicts.
//
// Against the form before (radix-2 stages across the 32 lanes of a warp,
// two real rows per complex row, accumulators in shared memory) a transform
// takes half the instructions and two thirds of the shared-memory passes.
//
// Per iteration: the forward kernel (per tile: x^ once, then per pair of
// exposures z, w_t = u_t z_t to the w planes) and the adjoint kernel (per
// tile: the sum over pairs, one inverse transform, the update of Eq. (2)). Work
// items are (tile, group of exposures): images with fewer tiles than SMs
// split the exposures into groups (fft_groups), whose accumulators the last
// CTA of a tile adds in group order. For r = 1 Gaussian with at least as many
// tiles as SMs the split forms run one persistent CTA per SM: whole waves of
// tiles, then the last wave's tiles cut into exposure ranges across all CTAs.
#include <math.h>

#include <algorithm>

#include "emd_corr.cuh"
#include "emd_fft.cuh"
#include "emd_internal.cuh"

namespace emd {
namespace {

constexpr int kFT = 128;                 // tile side
constexpr int kFP = 130;                 // row pitch in shared memory (complex)
constexpr int kFBuf = kFT * kFP;         // float2 of the transform buffer
constexpr int kFThreads = 512;           // 64 groups of eight lanes
constexpr int kSlots = 64 * kFT;         // float2 of the 64 column slots
constexpr int kCol = kSlots + kFT;       // the slots, then column 64
constexpr int kPairSpec = 2 * kSlots;    // S1, then S2 (slot 0 of S2: column 64)
constexpr float kFScale = 1.0f / (kFT * kFT);
constexpr int kSMs = 152;

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {  // a conj(b)
  return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// a + b conj(c)
__device__ __forceinline__ float2 cfmac(float2 a, float2 b, float2 c) {
  a.x = fmaf(b.x, c.x, a.x);
  a.y = fmaf(b.y, c.x, a.y);
  a.x = fmaf(b.y, c.y, a.x);
  a.y = fmaf(-b.x, c.y, a.y);
  return a;
}
// a + b c
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
  a.x = fmaf(b.x, c.x, a.x);
  a.y = fmaf(b.x, c.y, a.y);
  a.x = fmaf(-b.y, c.y, a.x);
  a.y = fmaf(b.y, c.x, a.y);
  return a;
}

// ---------------------------------------------------------------------------
// DFTs in registers (INV: conjugate twiddles, unscaled)
// ---------------------------------------------------------------------------

// a * exp(-+ i pi / 2)
template <bool INV>
__device__ __forceinline__ float2 rot(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <bool INV>
__device__ __forceinline__ void dft4(float2& a, float2& b, float2& c, float2& d) {
  const float2 s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(b, d), s3 = rot<INV>(csub(b, d));
  a = cadd(s0, s2);
  b = cadd(s1, s3);
  c = csub(s0, s2);
  d = csub(s1, s3);
}

// a * (wr -+ i wi): wr, wi the cosine and sine of the (positive) angle
template <bool INV>
__device__ __forceinline__ float2 cmulk(float2 a, float wr, float wi) {
  return INV ? make_float2(a.x * wr - a.y * wi, a.y * wr + a.x * wi)
             : make_float2(a.x * wr + a.y * wi, a.y * wr - a.x * wi);
}

constexpr float kR2 = 0.70710678118654752440f;   // cos(pi/4)
constexpr float kC8 = 0.92387953251128675613f;   // cos(pi/8)
constexpr float kS8 = 0.38268343236508977173f;   // sin(pi/8)

// eight points at v[0], v[1], ..., natural in and out
template <bool INV>
__device__ __forceinline__ void dft8(float2* v) {
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<INV>(e0, e1, e2, e3);
  dft4<INV>(o0, o1, o2, o3);
  // o1 w, o2 w^2, o3 w^3 with w = exp(-+ i pi / 4)
  o1 = INV ? make_float2(kR2 * (o1.x - o1.y), kR2 * (o1.x + o1.y))
           : make_float2(kR2 * (o1.x + o1.y), kR2 * (o1.y - o1.x));
  o2 = rot<INV>(o2);
  o3 = INV ? make_float2(-kR2 * (o3.x + o3.y), kR2 * (o3.x - o3.y))
           : make_float2(kR2 * (o3.y - o3.x), -kR2 * (o3.x + o3.y));
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1);
  v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2);
  v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3);
  v[7] = csub(e3, o3);
}

// sixteen points, natural in and out
template <bool INV>
__device__ __forceinline__ void dft16(float2 (&v)[16]) {
#pragma unroll
  for (int b = 0; b < 4; ++b) dft4<INV>(v[b], v[4 + b], v[8 + b], v[12 + b]);  // v[4 k + b]: y_b[k]
  v[5] = cmulk<INV>(v[5], kC8, kS8);                                      // w^1
  v[6] = INV ? make_float2(kR2 * (v[6].x - v[6].y), kR2 * (v[6].x + v[6].y))
             : make_float2(kR2 * (v[6].x + v[6].y), kR2 * (v[6].y - v[6].x));  // w^2
  v[7] = cmulk<INV>(v[7], kS8, kC8);                                      // w^3
  v[9] = INV ? make_float2(kR2 * (v[9].x - v[9].y), kR2 * (v[9].x + v[9].y))
             : make_float2(kR2 * (v[9].x + v[9].y), kR2 * (v[9].y - v[9].x));  // w^2
  v[10] = rot<INV>(v[10]);                                                // w^4
  v[11] = INV ? make_float2(-kR2 * (v[11].x + v[11].y), kR2 * (v[11].x - v[11].y))
              : make_float2(kR2 * (v[11].y - v[11].x), -kR2 * (v[11].x + v[11].y));  // w^6
  v[13] = cmulk<INV>(v[13], kS8, kC8);                                    // w^3
  v[14] = INV ? make_float2(-kR2 * (v[14].x + v[14].y), kR2 * (v[14].x - v[14].y))
              : make_float2(kR2 * (v[14].y - v[14].x), -kR2 * (v[14].x + v[14].y));  // w^6
  v[15] = cmulk<INV>(v[15], -kC8, -kS8);                                  // w^9
#pragma unroll
  for (int k = 0; k < 4; ++k) dft4<INV>(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
  // v[4 k1 + k2] holds X[k1 + 4 k2]: transpose the register names
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = a + 1; b < 4; ++b) {
      const float2 t = v[4 * a + b];
      v[4 * a + b] = v[4 * b + a];
      v[4 * b + a] = t;
    }
}

// (exp(-2 pi i j 2k / 128), exp(-2 pi i j (2k + 1) / 128)) at tw[8 k + j]
__device__ __forceinline__ void init_twiddles(float4* tw) {
  for (int e = threadIdx.x; e < kFT / 2; e += blockDim.x) {
    const int j = e & 7, k = e >> 3;
    float s0, c0, s1, c1;
    sincospif((float)(2 * k * j) / 64.f, &s0, &c0);
    sincospif((float)((2 * k + 1) * j) / 64.f, &s1, &c1);
    tw[e] = make_float4(c0, -s0, c1, -s1);
  }
  __syncthreads();
}
__device__ __forceinline__ void twiddle(float2 (&v)[16], const float4* tw, int t) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float4 w = tw[8 * k + t];
    if (k) v[2 * k] = cmul(v[2 * k], make_float2(w.x, w.y));
    v[2 * k + 1] = cmul(v[2 * k + 1], make_float2(w.z, w.w));
  }
}
__device__ __forceinline__ void twiddle_conj(float2 (&v)[16], const float4* tw, int t) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float4 w = tw[8 * k + t];
    if (k) v[2 * k] = cmulc(v[2 * k], make_float2(w.x, w.y));
    v[2 * k + 1] = cmulc(v[2 * k + 1], make_float2(w.z, w.w));
  }
}

// Launches of small grids are programmatic dependents of each other
// (launch_dependent): the next kernel's CTAs are set up on free SMs while this
// one runs, and wait here for it to complete before they read anything it wrote.
__device__ __forceinline__ void after_previous_launch() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

struct Lane {
  int warp, grp, t;  // warp, group of eight lanes in it, lane in the group
  __device__ Lane() : warp(threadIdx.x >> 5), grp((threadIdx.x >> 3) & 3), t(threadIdx.x & 7) {}
  // row of group k of this warp in 32-row block blk: a half-warp's two rows are
  // 4 apart (distinct bank pairs: 4 pitches are 8 mod 16 complex)
  __device__ int row(int blk, int k) const {
    return 32 * blk + (warp & 3) + 8 * ((warp >> 2) & 1) + 4 * (k & 1) + 16 * (k >> 1);
  }
  __device__ int row(int blk) const { return row(blk, grp); }
  // column slot of this group: a half-warp's two columns (and partners) are adjacent
  __device__ int slot() const { return 4 * warp + grp; }
};

// 128-point transforms of one line of the buffer by a group of eight lanes, the
// line's own storage carrying the exchange. Forward: v[i] = element t + 8 i in;
// out v[q] = frequency 2 t + 16 q, v[8 + q] = 2 t + 1 + 16 q. Inverse
// (unscaled): the reverse.
//
// Rows (element e at base + e, 16-byte aligned): the two frequencies of a lane
// travel as one 16-byte word, word 8 k + (j ^ k) holding frequencies 2 k and
// 2 k + 1 of lane j's 16-point DFT.
__device__ __forceinline__ void fft_row(float2 (&v)[16], float2* base, const float4* tw, int t) {
  dft16<false>(v);
  twiddle(v, tw, t);
  float4* b4 = reinterpret_cast<float4*>(base);
  __syncwarp();  // the group has read its inputs from the line
#pragma unroll
  for (int k = 0; k < 8; ++k)
    b4[8 * k + (t ^ k)] = make_float4(v[2 * k].x, v[2 * k].y, v[2 * k + 1].x, v[2 * k + 1].y);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float4 w = b4[8 * t + (t ^ j)];
    v[j] = make_float2(w.x, w.y);
    v[8 + j] = make_float2(w.z, w.w);
  }
  dft8<false>(v);
  dft8<false>(v + 8);
}
__device__ __forceinline__ void ifft_row(float2 (&v)[16], float2* base, const float4* tw, int t) {
  dft8<true>(v);
  dft8<true>(v + 8);
  float4* b4 = reinterpret_cast<float4*>(base);
  __syncwarp();  // the group has read its inputs from the line
#pragma unroll
  for (int j = 0; j < 8; ++j)
    b4[8 * t + (t ^ j)] = make_float4(v[j].x, v[j].y, v[8 + j].x, v[8 + j].y);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float4 w = b4[8 * k + (t ^ k)];
    v[2 * k] = make_float2(w.x, w.y);
    v[2 * k + 1] = make_float2(w.z, w.w);
  }
  twiddle_conj(v, tw, t);
  dft16<true>(v);
}

// Columns (element e at base + e kFP): frequency p of lane j's 16-point DFT at
// element 8 p + (j ^ (p / 2)).
__device__ __forceinline__ void fft_col(float2 (&v)[16], float2* base, const float4* tw, int t) {
  dft16<false>(v);
  twiddle(v, tw, t);
  __syncwarp();  // the group has read its inputs from the line
#pragma unroll
  for (int p = 0; p < 16; ++p) base[(8 * p + (t ^ (p >> 1))) * kFP] = v[p];
  __syncwarp();
  float2* mine = base + 16 * t * kFP;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    v[j] = mine[(t ^ j) * kFP];
    v[8 + j] = mine[(8 + (t ^ j)) * kFP];
  }
  dft8<false>(v);
  dft8<false>(v + 8);
}
__device__ __forceinline__ void ifft_col(float2 (&v)[16], float2* base, const float4* tw, int t) {
  dft8<true>(v);
  dft8<true>(v + 8);
  __syncwarp();  // the group has read its inputs from the line
  float2* mine = base + 16 * t * kFP;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    mine[(t ^ j) * kFP] = v[j];
    mine[(8 + (t ^ j)) * kFP] = v[8 + j];
  }
  __syncwarp();
#pragma unroll
  for (int p = 0; p < 16; ++p) v[p] = base[(8 * p + (t ^ (p >> 1))) * kFP];
  twiddle_conj(v, tw, t);
  dft16<true>(v);
}

// frequencies of a row to and from its natural positions
__device__ __forceinline__ void store_freqs(float2* row, const float2 (&v)[16], int t) {
  float4* b4 = reinterpret_cast<float4*>(row);
  __syncwarp();  // the group's exchange reads of this row are done
#pragma unroll
  for (int q = 0; q < 8; ++q) b4[t + 8 * q] = make_float4(v[q].x, v[q].y, v[8 + q].x, v[8 + q].y);
}
__device__ __forceinline__ void load_freqs(const float2* row, float2 (&v)[16], int t) {
  const float4* b4 = reinterpret_cast<const float4*>(row);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 w = b4[t + 8 * q];
    v[q] = make_float2(w.x, w.y);
    v[8 + q] = make_float2(w.z, w.w);
  }
}
// elements t + 8 i of a column
__device__ __forceinline__ void load_col(const float2* col, float2 (&v)[16], int t, bool conj) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v[i] = col[(t + 8 * i) * kFP];
    if (conj) v[i].y = -v[i].y;
  }
}
__device__ __forceinline__ void store_col(float2* col, const float2 (&v)[16], int t, bool conj) {
  __syncwarp();  // the group's exchange reads of this column are done
#pragma unroll
  for (int i = 0; i < 16; ++i)
    col[(t + 8 * i) * kFP] = conj ? make_float2(v[i].x, -v[i].y) : v[i];
}

// the same where not every group of the warp stores
__device__ __forceinline__ void store_col_group(float2* col, const float2 (&v)[16], const Lane& L,
                                                bool conj) {
  __syncwarp(0xffu << (8 * L.grp));
#pragma unroll
  for (int i = 0; i < 16; ++i)
    col[(L.t + 8 * i) * kFP] = conj ? make_float2(v[i].x, -v[i].y) : v[i];
}

// This thread's 16 values of its column slot in a slot array: v at
// (warp 16 + v) 32 + lane (a warp's loads are contiguous)
__device__ __forceinline__ int slot_off() { return (threadIdx.x >> 5) * 512 + (threadIdx.x & 31); }
__device__ __forceinline__ void store_slot(float2* a, const float2 (&v)[16]) {
  a += slot_off();
#pragma unroll
  for (int i = 0; i < 16; ++i) a[32 * i] = v[i];
}

// The same slice through shared memory: a warp copies its contiguous 4 KB of a
// slot array (or of S2) to its own staging buffer, one step before it is
// needed, so that the L2 latency passes during the transform between. Each
// warp waits for its own copies only.
constexpr int kStage = 512;  // float2 per warp
__device__ __forceinline__ void stage_slot(float2* st, const float2* a) {
  const int lane = threadIdx.x & 31;
  const float2* src = a + (threadIdx.x >> 5) * 512 + 2 * lane;
  const unsigned dst = (unsigned)__cvta_generic_to_shared(st + 2 * lane);
  __syncwarp();  // the warp's reads of the previous slice are done
#pragma unroll
  for (int k = 0; k < 8; ++k)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 * k), "l"(src + 64 * k)
                 : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void staged_ready() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
}

// L2 prefetch by the whole CTA, one 128-byte line per lane: `rows` rows of
// `bytes` bytes, `pitch` bytes apart (a tile's data of the next pair, which
// DRAM would else deliver late). Bulk prefetches, one per row from one warp,
// held that warp up for longer than they saved.
__device__ __forceinline__ void prefetch_rows(const void* base, long long pitch, int rows,
                                              int bytes) {
  const int lines = (bytes + 254) >> 7;  // whatever the row's offset in its first line
  for (int e = threadIdx.x; e < rows * lines; e += kFThreads) {
    const int r = e / lines, l = e - r * lines;
    const char* p = static_cast<const char*>(base) + r * pitch + min(128 * l, bytes - 1);
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
  }
}

// the 128 x 128 region with origin (r0, c0) of a padded plane of `size`-byte elements
__device__ __forceinline__ void prefetch_region(const void* plane, int size, const Geom& g, int r0,
                                                int c0) {
  const int ra = max(r0, 0), rb = min(r0 + kFT, g.H), ca = max(c0, 0), cb = min(c0 + kFT, g.W);
  prefetch_rows(static_cast<const char*>(plane) + ((long long)(g.B + ra) * g.P + g.B + ca) * size,
                (long long)size * g.P, rb - ra, size * (cb - ca));
}

// The second column of a slot: 128 - m (through the conjugate), or 64 for slot 0.
__device__ __forceinline__ int second_col(int m) { return m ? kFT - m : 64; }

// Row transforms of the 128 x 128 region whose rows load(r, t, v) gives
// (v[i] = element t + 8 i of row r); ends at a CTA barrier
template <class Load>
__device__ __forceinline__ void rows_forward(float2* buf, const float4* tw, const Lane& L,
                                             Load&& load) {
#pragma unroll 1
  for (int round = 0; round < 2; ++round) {
    const int r = L.row((L.warp >> 3) + 2 * round);
    float2 v[16];
    load(r, v);
    fft_row(v, buf + r * kFP, tw, L.t);
    store_freqs(buf + r * kFP, v, L.t);
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// tensor memory as thread-private storage (r = 2)
// ---------------------------------------------------------------------------

// A slot's spectrum is 16 complex values a thread, so four phases' are 128
// words of each of the 512 threads: the SM's 256 KB of tensor memory, which
// the FFT form does not use otherwise. x^ (forward) and the Gaussian
// accumulators (adjoint) of r = 2 live there instead of in a per-tile scratch
// in L2, whose read-modify-write per pair and phase left the adjoint waiting
// (issue slots 16 % busy, now 39 %: 33 x 1024^2, K = 85: forward 339 -> 245 us,
// adjoint 791 -> 319 us).
constexpr int kTmPhases = 4;
constexpr int kTmCols = 512;  // all columns; thread: lane tid mod 128, 128 columns

// All warps of the CTA; one CTA per SM (shared memory), so the allocation does
// not wait.
__device__ __forceinline__ uint32_t tmem_begin(uint32_t* base_s) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(base_s)),
                 "r"(kTmCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t warp = threadIdx.x >> 5;
  return *base_s + ((warp & 3) << 21) + (warp >> 2) * (kTmPhases * 32);
}
__device__ __forceinline__ void tmem_end(uint32_t base) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base),
                 "r"(kTmCols));
  }
}
// this thread's 16 values of one phase (whole warps, converged)
__device__ __forceinline__ void tmem_load(float2 (&v)[16], uint32_t addr) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
        "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
        "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
        "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
        "=r"(r[30]), "=r"(r[31])
      : "r"(addr)
      : "memory");
  // (the operands order every use of the values after the wait)
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]),
                 "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]),
                 "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]),
                 "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]),
                 "+r"(r[31])
               :
               : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i)
    v[i] = make_float2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
}
__device__ __forceinline__ void tmem_store(uint32_t addr, const float2 (&v)[16]) {
  uint32_t r[32];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    r[2 * i] = __float_as_uint(v[i].x);
    r[2 * i + 1] = __float_as_uint(v[i].y);
  }
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(addr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]),
      "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]),
      "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]),
      "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// spectra of the kernels
// ---------------------------------------------------------------------------

// 1 / s_t of exposure blockIdx.x: the power of two nearest, in logarithm, to the sum
// of its |taps| (of one of R2 phases on average: 1 for a PSF of unit sum)
__global__ void __launch_bounds__(256)
    fft_scale_kernel(const float* __restrict__ ka, int taps, int R2,
                     float* __restrict__ inv_scale) {
  __shared__ double red[8];
  const float* k = ka + (long long)blockIdx.x * R2 * taps;
  double v = 0.0;
  for (int e = threadIdx.x; e < R2 * taps; e += blockDim.x) v += fabs((double)k[e]);
  const double sum = block_sum_f64(v, red);
  if (threadIdx.x == 0) {
    const bool ok = sum > 0.0 && isfinite(sum);  // no taps, or none that are numbers
    const int e = ok ? max(-40, min(40, ilogb(sum / R2 * 1.4142135623730951))) : 0;
    inv_scale[blockIdx.x] = exp2f((float)e);
  }
}

// inv_scale[n]: whether any is not 1 (only then the forward pass loads and multiplies
// by them, 1 to 2 % of its time)
__global__ void __launch_bounds__(256) fft_scaled_kernel(int n, float* __restrict__ inv_scale) {
  bool any = false;
  for (int t = threadIdx.x; t < n; t += blockDim.x) any |= inv_scale[t] != 1.f;
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) inv_scale[n] = any ? 1.f : 0.f;
}

// One CTA per (pair, phase): S1 and S2 of k_a + i k_b; single = true: per
// (exposure, phase) the slots and column 64 of k_t alone. The Kc x Kc phase
// kernels (row pitch KP; for r = 1 the PSFs) at the top-left of a zero tile.
__global__ void __launch_bounds__(kFThreads, 1)
    fft_spectra_kernel(const float* __restrict__ ka, const float* __restrict__ inv_scale, int n,
                       int R2, int Kc, int KP, bool single, float2* __restrict__ out) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  init_twiddles(tw);
  const Lane L;
  const int q = blockIdx.x / R2, phi = blockIdx.x - q * R2;
  const int ta = single ? q : 2 * q, tb = ta + 1;
  const float* fa = ka + ((long long)ta * R2 + phi) * Kc * KP;
  const float* fb = !single && tb < n ? ka + ((long long)tb * R2 + phi) * Kc * KP : nullptr;
  // with the inverse transform's 1 / 128^2, exact as well
  const float sa = single ? kFScale : kFScale / inv_scale[ta];
  const float sb = fb ? kFScale / inv_scale[tb] : 1.f;
  rows_forward(fsm, tw, L, [&](int r, float2 (&v)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int c = L.t + 8 * i;
      const bool in = r < Kc && c < Kc;
      v[i] = make_float2(in ? sa * fa[r * KP + c] : 0.f, in && fb ? sb * fb[r * KP + c] : 0.f);
    }
  });
  const int m = L.slot();
  out += (long long)blockIdx.x * (single ? kCol : kPairSpec);
  float2 v[16];
  load_col(fsm + m, v, L.t, false);
  fft_col(v, fsm + m, tw, L.t);
  store_slot(out, v);
  const int m2 = second_col(m);
  load_col(fsm + m2, v, L.t, m != 0);
  fft_col(v, fsm + m2, tw, L.t);
  if (!single) {
    store_slot(out + kSlots, v);
  } else if (m == 0) {
#pragma unroll
    for (int i = 0; i < 16; ++i) out[kSlots + 8 * i + L.t] = v[i];
  }
}

// ---------------------------------------------------------------------------
// forward model
// ---------------------------------------------------------------------------

// x^ of one phase: the slot of this thread into X, column 64 into x64 (128
// entries); starts and ends at a CTA barrier
__device__ __forceinline__ void region_spectrum(const float* plane, const Geom& g, int r0, int c0,
                                                float2* buf, const float4* tw, const Lane& L,
                                                float2 (&X)[16], float2* x64) {
  rows_forward(buf, tw, L, [&](int r, float2 (&v)[16]) {
    const int i = r0 + r;
    const bool row_in = i >= 0 && i < g.H;
    const float* src = plane + (long long)(g.B + i) * g.P + g.B;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int j = c0 + L.t + 8 * q;
      v[q] = make_float2(row_in && j >= 0 && j < g.W ? __ldcg(src + j) : 0.f, 0.f);
    }
  });
  // column 64 first (slot 0's group, and with it its warp, for the warp
  // barriers), then the slots: one copy of the transform's code
  const int m = L.slot();
#pragma unroll 1
  for (int h = L.warp == 0; h >= 0; --h) {
    float2* col = buf + (h ? second_col(m) : m);
    load_col(col, X, L.t, false);
    fft_col(X, col, tw, L.t);
    if (h && m == 0) {
#pragma unroll
      for (int i = 0; i < 16; ++i) x64[8 * i + L.t] = X[i];
    }
  }
  __syncthreads();
}

// The forward pass of one tile for the pairs of exposures [q0, q1). R1: r = 1
// (x^ in registers; otherwise the phases' x^ in xs). Starts and ends at a CTA
// barrier, so a persistent CTA can run many; (nty, ntx), if known, is the tile
// it runs next, whose x region is brought into L2 meanwhile. TM: r = 2 with
// the phases' x^ in tensor memory (tm) and x64 of four phases.
template <bool R1, bool STUDENT, bool TM = false>
__device__ void fft_forward_tile(const Shape& s, const FftLaunch& a, int ty, int tx, float2* xs,
                                 float2* buf, float2* x64, const float4* tw, int q0, int q1,
                                 int nty = -1, int ntx = 0, uint32_t tm = 0) {
  const Geom& g = s.g;
  const Lane L;
  const int hc = s.hc, B = kFT - 2 * hc, R2 = TM ? kTmPhases : s.R2;
  const int i0 = ty * B, j0 = tx * B;
  const int m = L.slot(), m2 = second_col(m);
  const int pmax = min(B, g.H - i0), qmax = min(B, g.W - j0);
  float2* st = buf + kFBuf + L.warp * kStage;
  const bool scaled = __ldg(a.inv_scale + s.n) != 0.f;  // some s_t is not 1
  auto prefetch_pair = [&](int q) {  // u (and y) of the tile
    for (int t = 2 * q; t < min(2 * q + 2, s.n); ++t) {
      const long long off = (long long)t * g.plane + (long long)(g.B + i0) * g.P + g.B + j0;
      prefetch_rows(a.u + off, 4LL * g.P, pmax, 4 * qmax);
      if (STUDENT) prefetch_rows(a.y + off, 4LL * g.P, pmax, 4 * qmax);
    }
  };
  prefetch_pair(q0);
  if (R1 || TM) stage_slot(st, a.spec + (long long)q0 * R2 * kPairSpec);
  float2 X[16];
  if (R1) {
    region_spectrum(a.x, g, i0 - hc, j0 - hc, buf, tw, L, X, x64);
  } else if (TM) {
#pragma unroll 1
    for (int ph = 0; ph < kTmPhases; ++ph) {
      region_spectrum(a.x + (long long)ph * g.plane, g, i0 - hc, j0 - hc, buf, tw, L, X,
                      x64 + ph * kFT);
      tmem_store(tm + 32 * ph, X);
    }
  } else {
    for (int ph = 0; ph < R2; ++ph) {
      region_spectrum(a.x + (long long)ph * g.plane, g, i0 - hc, j0 - hc, buf, tw, L, X,
                      xs + (long long)ph * kCol + kSlots);
      store_slot(xs + (long long)ph * kCol, X);
    }
  }
  for (int q = q0; q < q1; ++q) {
    const float2* S = a.spec + (long long)q * R2 * kPairSpec;
    if (q + 1 < q1)
      prefetch_pair(q + 1);
    else if (nty >= 0)
      prefetch_region(a.x, 4, g, nty * B - hc, ntx * B - hc);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {  // column m, then its partner
      float2 v[16];
      if (R1) {
        const float2* sp = st + (threadIdx.x & 31);
        staged_ready();
        if (h == 1 && m == 0) {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = cmul(x64[8 * i + L.t], sp[32 * i]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = cmul(X[i], sp[32 * i]);
        }
        // S2 arrives during this column's transform, the next pair's S1 during
        // the second column's and the rows
        if (h == 0)
          stage_slot(st, S + kSlots);
        else if (q + 1 < q1)
          stage_slot(st, S + kPairSpec);
      } else if (TM) {
        // S of phase 0 staged as for r = 1, the others' a phase ahead in registers
        const float2* sp = S + h * kSlots + slot_off();
        const bool c64 = h == 1 && m == 0;
        float2 kv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          kv[i] = __ldg(sp + kPairSpec + 32 * i);
          v[i] = make_float2(0.f, 0.f);
        }
        staged_ready();
        const float2* s0 = st + (threadIdx.x & 31);
#pragma unroll 1
        for (int ph = 0; ph < kTmPhases; ++ph) {
          float2 x[16];
          tmem_load(x, tm + 32 * ph);
          if (c64) {
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = x64[ph * kFT + 8 * i + L.t];
          }
          if (ph == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = cfma(v[i], x[i], s0[32 * i]);
            if (h == 0)
              stage_slot(st, S + kSlots);
            else if (q + 1 < q1)
              stage_slot(st, S + kTmPhases * kPairSpec);
          } else {
            sp += kPairSpec;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              v[i] = cfma(v[i], x[i], kv[i]);
              if (ph + 1 < kTmPhases) kv[i] = __ldg(sp + kPairSpec + 32 * i);
            }
          }
          __syncwarp();
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = make_float2(0.f, 0.f);
        const bool c64 = h == 1 && m == 0;
        const int xstep = c64 ? 8 : 32;
#pragma unroll 2
        for (int ph = 0; ph < R2; ++ph) {
          const float2* sp = S + (long long)ph * kPairSpec + h * kSlots + slot_off();
          const float2* xp = xs + (long long)ph * kCol + (c64 ? kSlots + L.t : slot_off());
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = cfma(v[i], xp[xstep * i], __ldg(sp + 32 * i));
        }
      }
      float2* col = buf + (h == 0 ? m : m2);
      ifft_col(v, col, tw, L.t);
      store_col(col, v, L.t, h == 1 && m != 0);
    }
    __syncthreads();
    // rows [2 hc, 128): z_a + i z_b at columns [2 hc, 128)
    const int ta = 2 * q, tb = min(ta + 1, s.n - 1);  // (an odd last exposure: z_b unused)
    const bool two = ta + 1 < s.n;
    const int c_lo = 2 * hc - L.t, c_hi = 2 * hc + qmax - L.t;  // columns t + 8 i: 8 i in [c_lo, c_hi)
#pragma unroll 1
    for (int blk = 3 - (L.warp >> 3); blk >= 0 && 32 * blk + 31 >= 2 * hc; blk -= 2) {
      const int r = L.row(blk), p = r - 2 * hc;
      const bool row_ok = p >= 0 && p < pmax;
      const long long rowoff = (long long)(g.B + i0 + p) * g.P + g.B + j0 - 2 * hc + L.t;
      const float* ua = a.u + (long long)ta * g.plane + rowoff;
      const float* ub = a.u + (long long)tb * g.plane + rowoff;
      float2 u[16];  // in flight during the transform
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const bool in = row_ok && 8 * i >= c_lo && 8 * i < c_hi;
        u[i] = make_float2(in ? __ldg(ua + 8 * i) : 0.f, in && two ? __ldg(ub + 8 * i) : 0.f);
      }
      // heavy-tailed: y of the first exposure also during the transform, of the
      // second during the first's weights (loads inside the loop below waited one
      // by one behind its stores: 1024^2 x 20, forward pass 277 -> 200 us)
      float yv[STUDENT ? 16 : 1];
      auto load_y = [&](float (&y)[STUDENT ? 16 : 1], int t) {
        const float* yp = a.y + (long long)t * g.plane + rowoff;
#pragma unroll
        for (int i = 0; i < 16; ++i)
          y[STUDENT ? i : 0] =
              row_ok && 8 * i >= c_lo && 8 * i < c_hi ? __ldg(yp + 8 * i) : 0.f;
      };
      if (STUDENT) load_y(yv, ta);
      float2 v[16];
      load_freqs(buf + r * kFP, v, L.t);
      ifft_row(v, buf + r * kFP, tw, L.t);
      if (!row_ok) continue;
      if (scaled) {  // z = v / s_t; the adjoint's source for the kernel s_t k_t is w / s_t
        const float ia = __ldg(a.inv_scale + ta), ib = __ldg(a.inv_scale + tb);
        const float fa = STUDENT ? ia : ia * ia, fb = STUDENT ? ib : ib * ib;
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = make_float2(v[i].x * fa, v[i].y * fb);
      }
      if (!STUDENT) {
        float2* w = a.w + (long long)q * g.plane + rowoff;
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (8 * i >= c_lo && 8 * i < c_hi)
            w[8 * i] = make_float2(u[i].x * v[i].x, u[i].y * v[i].y);
      } else {
        // heavy-tailed weights u' = u (nu+1) / (nu + u (y - z)^2): (u' z, u' y) per
        // exposure
        const float nu1 = a.nu + 1.f;
        float yb[STUDENT ? 16 : 1];
        load_y(yb, tb);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (e && !two) break;
          float2* w = a.w + (long long)(ta + e) * g.plane + rowoff;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            if (8 * i >= c_lo && 8 * i < c_hi) {
              const float z = e ? v[i].y : v[i].x, uv = e ? u[i].y : u[i].x;
              const float y = e ? yb[STUDENT ? i : 0] : yv[STUDENT ? i : 0];
              const float d = y - z;
              const float us = uv > 0.f ? uv * nu1 / fmaf(uv * d, d, a.nu) : 0.f;
              w[8 * i] = make_float2(us * z, us * y);
            }
          }
        }
      }
    }
    __syncthreads();  // the buffer is free for the next pair
  }
}

// ---------------------------------------------------------------------------
// adjoint and update
// ---------------------------------------------------------------------------

// one pixel of Eq. (2)
__device__ __forceinline__ float update_pixel(float xo, float d, float nraw, float nt) {
  // The transform leaves a rounding floor (~1e-7 of the tile's weighted
  // model) where the exact denominator is 0. The numerator is +0 exactly there,
  // where no valid pixel lies in the footprint, and nowhere else (a sum that
  // cancels is -0, numerator_marks_kernel): x then stays, as for Den = 0; with
  // Student-t weights too, since u' = 0 exactly where u = 0.
  float xv = xo;
  if (d > 0.f && __float_as_uint(nraw) != 0u) {
    const float nv = fmaxf(nt, 0.f);
    if (d < 1e-30f)  // denominator near zero: guarded ratio in FP64
      xv = (float)((double)xo * (double)nv / (double)d);
    else
      xv = xo * nv / d;
  }
  return xv;
}

// From the columns in the buffer (every column of every row): inverse row
// transforms of the rows [0, B) and the update of one phase. STUDENT: real part
// Den, imaginary part N' over inv_scale. Starts and ends at a CTA barrier.
template <bool STUDENT>
__device__ __forceinline__ void rows_update(const Shape& s, const FftLaunch& a, int phi, int i0,
                                            int j0, float2* buf, const float4* tw, const Lane& L,
                                            float inv_scale = 1.f) {
  const Geom& g = s.g;
  const int B = kFT - 2 * s.hc;
  const int pmax = min(B, g.H - i0), qmax = min(B, g.W - j0);
#pragma unroll 1
  for (int blk = L.warp >> 3; blk < 4 && 32 * blk < pmax; blk += 2) {
    const int r = L.row(blk);
    const long long off =
        (long long)phi * g.plane + (long long)(g.B + i0 + r) * g.P + g.B + j0 + L.t;
    float xo[16], nraw[16];  // in flight during the transform
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const bool in = r < pmax && L.t + 8 * i < qmax;
      xo[i] = in ? __ldcg(a.x + off + 8 * i) : 0.f;
      nraw[i] = in ? __ldg(a.N + off + 8 * i) : 0.f;
    }
    float2 v[16];
    load_freqs(buf + r * kFP, v, L.t);
    ifft_row(v, buf + r * kFP, tw, L.t);
    if (r >= pmax) continue;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (L.t + 8 * i < qmax)
        a.xn[off + 8 * i] =
            update_pixel(xo[i], v[i].x, nraw[i], STUDENT ? v[i].y * inv_scale : nraw[i]);
  }
  __syncthreads();
}

// Gaussian: the Hermitian accumulator of this thread's slot (acc) and, for
// slot 0, column 64 (a64, 128 entries) -> the buffer's columns. H counts m >= 1
// twice (see the file comment); columns 0 and 64 keep the real part.
__device__ __forceinline__ void columns_gauss(const float2 (&acc)[16], const float2* a64, float2* buf,
                                              const float4* tw, const Lane& L) {
  const int m = L.slot(), m2 = second_col(m);
  const float sc = m ? 0.5f : 1.f;
  // column 64 first (slot 0's group, and with it its warp, for the warp
  // barriers), then the slots: one copy of the transform's code
#pragma unroll 1
  for (int h = L.warp == 0; h >= 0; --h) {
    float2 v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      v[i] = acc[i];
      if (h) v[i] = m ? make_float2(0.f, 0.f) : a64[8 * i + L.t];
    }
    float2* col = buf + (h ? m2 : m);
    ifft_col(v, col, tw, L.t);
    if (h && m) continue;  // (only slot 0's second column is wanted)
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = make_float2(sc * v[i].x, m ? sc * v[i].y : 0.f);
    store_col_group(col, v, L, false);
    if (m) store_col_group(buf + m2, v, L, true);
  }
  __syncthreads();
}

// Student-t: the slot's two columns, m from f and 128 - m (64 for slot 0) from
// the conjugate of g -> the buffer's columns
__device__ __forceinline__ void columns_student(float2 (&f)[16], const float2 (&gv)[16], float2* buf,
                                                const float4* tw, const Lane& L) {
  const int m = L.slot(), m2 = second_col(m);
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    float2* col = buf + (h ? m2 : m);
    if (h) {
#pragma unroll
      for (int i = 0; i < 16; ++i) f[i] = gv[i];
    }
    ifft_col(f, col, tw, L.t);
    store_col(col, f, L.t, h && m != 0);
  }
  __syncthreads();
}

// A warp's four rows (L.row(blk)) of the w region with origin (r0, c0) of
// plane `w` (float2 on the padded planes; zero outside the image), by
// asynchronous copies to dst, row pitch kFP: 32 lanes copy 256 contiguous
// bytes, where loads in the transform's own order (eight lanes a row) touch
// four rows an instruction.
__device__ __forceinline__ void copy_w(float2* dst, const float2* w, const Geom& g, int r0, int c0,
                                       int blk, const Lane& L) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = L.row(blk, k), i = r0 + r;
    const bool row_in = i >= 0 && i < g.H;
    const float2* src = w + (long long)(g.B + (row_in ? i : 0)) * g.P + g.B;
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst + L.row(0, k) * kFP + lane);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = c0 + lane + 32 * q;
      const bool in = row_in && j >= 0 && j < g.W;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d + 256 * q),
                   "l"(src + (in ? j : 0)), "r"(in ? 8 : 0)
                   : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void copies_ready() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
}

// Heavy-tailed adjoint: the power of two that brings w2 = u' y to the size of
// w = u' z on the tile's region with origin (r0, c0), from the largest |w| and |w2| of
// every fourth row of the first exposure that has any (all exposures see one sky).
// Every group of a tile takes the same one. Called by the whole CTA.
__device__ float student_scale(const FftLaunch& a, const Geom& g, int n, int r0, int c0) {
  __shared__ unsigned peak[2];
  float scale = 1.f;
  for (int t = 0; t < n; ++t) {
    __syncthreads();  // the last readers of the peaks are done
    if (threadIdx.x < 2) peak[threadIdx.x] = 0u;
    __syncthreads();
    const float2* w = a.w + (long long)t * g.plane + (long long)g.B * g.P + g.B;
    float m1 = 0.f, m2 = 0.f;
#pragma unroll
    for (int k = 0; k < kFT * kFT / 4 / kFThreads; ++k) {
      const int e = threadIdx.x + k * kFThreads, i = r0 + 4 * (e / kFT), j = c0 + e % kFT;
      if (i >= 0 && i < g.H && j >= 0 && j < g.W) {
        const float2 v = __ldcg(w + (long long)i * g.P + j);
        m1 = fmaxf(m1, fabsf(v.x));
        m2 = fmaxf(m2, fabsf(v.y));
      }
    }
    // (values >= 0: ordered as their bits)
    m1 = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m1)));
    m2 = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m2)));
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&peak[0], __float_as_uint(m1));
      atomicMax(&peak[1], __float_as_uint(m2));
    }
    __syncthreads();
    const float p1 = __uint_as_float(peak[0]), p2 = __uint_as_float(peak[1]);
    if (p1 > 0.f && p2 > 0.f) {
      if (isfinite(p1) && isfinite(p2))
        scale = exp2f((float)max(-60, min(60, ilogbf(p1) - ilogbf(p2))));
      break;
    }
  }
  return scale;
}

// Row transforms of a w region. The warp's rows of the blocks 0 and 1 are
// in flight to or in its part of the staging buffer (copy_w a column phase
// ago), or, stage null, in flight to their place in buf; those of the blocks
// 2 and 3 come straight to their place during the first transforms. STUDENT: the
// second image times scale. Ends at a CTA barrier.
template <bool STUDENT>
__device__ __forceinline__ void w_rows(float2* stage, const float2* w, const Geom& g, int r0,
                                       int c0, float2* buf, const float4* tw, const Lane& L,
                                       float scale = 1.f) {
  const int blk = L.warp >> 3;
  copies_ready();
  copy_w(buf + (blk + 2) * 32 * kFP, w, g, r0, c0, blk + 2, L);
#pragma unroll 1
  for (int round = 0; round < 2; ++round) {
    const int r = L.row(blk + 2 * round);
    const float2* src = (round || !stage ? buf : stage) + r * kFP;
    if (round) copies_ready();
    float2 v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      v[i] = src[L.t + 8 * i];
      if (STUDENT) v[i].y *= scale;
    }
    fft_row(v, buf + r * kFP, tw, L.t);
    store_freqs(buf + r * kFP, v, L.t);
  }
  __syncthreads();
}

constexpr unsigned kPartPolls = 1u << 23;  // x ~0.3 us per poll: seconds, not a hang

// A tile cut into parts (consecutive pairs) on different CTAs of a split
// launch: part i > 0 waits (bounded) for the tile's flag to reach i, starts
// from the accumulator part i - 1 left in its CTA's slot, and, unless it is
// the last part, leaves its own in this CTA's slot and raises the flag to
// i + 1; the last part finishes the tile and resets the flag. The pairs are
// summed in the order a whole-tile CTA sums them (the same bits). A wait that
// gives up sets the timeout bit of the error word and starts from zero.
__device__ void publish_part(const FftLaunch& a, int tile, const float2 (&acc)[16],
                             const float2* a64, int part) {
  float2* slot = a.partials + (long long)blockIdx.x * kCol;
  store_slot(slot, acc);
  for (int e = threadIdx.x; e < kFT; e += blockDim.x) slot[kSlots + e] = a64[e];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) st_release(a.counters + tile, part + 1);
}

__device__ void resume_part(const FftLaunch& a, int tile, float2 (&acc)[16], float2* a64, int part,
                            int prev_cta, bool last) {
  __shared__ int ok;
  if (threadIdx.x == 0) {
    unsigned i = 0;
    while (i < kPartPolls && ld_acquire(a.counters + tile) < part) {
      __nanosleep(200);
      ++i;
    }
    ok = i < kPartPolls;
    if (!ok)
      atomicOr(a.err, kErrTimeout);
    else if (last)
      a.counters[tile] = 0;  // ready for the next launch
  }
  __syncthreads();
  const float2* slot = a.partials + (long long)prev_cta * kCol;
  const float2* mine = slot + slot_off();
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = ok ? __ldcg(mine + 32 * i) : make_float2(0.f, 0.f);
  for (int e = threadIdx.x; e < kFT; e += blockDim.x)
    a64[e] = ok ? __ldcg(slot + kSlots + e) : make_float2(0.f, 0.f);
  __syncthreads();
}

// groups > 1: counts this CTA's group of the tile in; the CTA that brings the
// last one returns true, with the others' accumulators visible to it, and the
// counter back at zero.
__device__ bool last_group(const FftLaunch& a, int tile) {
  __shared__ int last_s;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool last = atomicAdd(a.counters + tile, 1) == a.groups - 1;
    if (last) a.counters[tile] = 0;
    last_s = last;
  }
  __syncthreads();
  if (last_s) __threadfence();
  return last_s != 0;
}

// The adjoint pass and the update of one tile, r = 1: the sources of the pairs
// [q0, q1) (Student-t: their exposures, w + i w2 each, into the accumulators of
// both columns of a slot). grp >= 0: group grp of the tile's groups (its
// accumulators go to partials; the last to arrive adds them and finishes).
// Otherwise (Gaussian) part `part` of a split launch (prev_cta < 0: from zero),
// which finishes the tile if it is the last. (nty, ntx): as in
// fft_forward_tile. Starts and ends at a CTA barrier.
template <bool STUDENT>
__device__ void fft_adjoint_tile(const Shape& s, const FftLaunch& a, int ty, int tx, int tile,
                                 float2* buf, float2* a64, const float4* tw, int q0, int q1,
                                 int grp, int part = 0, int prev_cta = -1, bool last = true,
                                 int nty = -1, int ntx = 0) {
  constexpr int kPer = STUDENT ? 2 * kSlots : kCol;  // float2 of a partial accumulator
  const Geom& g = s.g;
  const Lane L;
  const int hc = s.hc, B = kFT - 2 * hc;
  const int i0 = ty * B, j0 = tx * B;
  const int m = L.slot(), m2 = second_col(m);
  const int blk = L.warp >> 3;
  float2 acc[16], acc2[STUDENT ? 16 : 1];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    acc[i] = make_float2(0.f, 0.f);
    if (STUDENT) acc2[STUDENT ? i : 0] = make_float2(0.f, 0.f);
  }
  if (!STUDENT) {
    if (prev_cta >= 0) {
      resume_part(a, tile, acc, a64, part, prev_cta, last);
    } else {
      for (int e = threadIdx.x; e < kFT; e += blockDim.x) a64[e] = make_float2(0.f, 0.f);
      __syncthreads();
    }
  }
  const int k0 = STUDENT ? 2 * q0 : q0, k1 = STUDENT ? min(2 * q1, s.n) : q1;
  const float scale = STUDENT ? student_scale(a, g, s.n, i0 - hc, j0 - hc) : 1.f;
  float2* stage = buf + kFBuf;
  float2* st = stage + L.warp * kStage;  // Student-t: this warp's slice of the spectrum
  if (!STUDENT)
    copy_w(stage + blk * 32 * kFP, a.w + (long long)k0 * g.plane, g, i0 - hc, j0 - hc, blk, L);
  for (int k = k0; k < k1; ++k) {
    const float2* w = a.w + (long long)k * g.plane;
    if (k + 1 < k1) {
      prefetch_region(w + g.plane, 8, g, i0 - hc, j0 - hc);
    } else {
      if (last) {  // what the update reads
        const long long off = (long long)(g.B + i0) * g.P + g.B + j0;
        const int rows = min(B, g.H - i0), bytes = 4 * min(B, g.W - j0);
        prefetch_rows(a.x + off, 4LL * g.P, rows, bytes);
        prefetch_rows(a.N + off, 4LL * g.P, rows, bytes);
      }
      if (nty >= 0) prefetch_region(a.w, 8, g, nty * B - hc, ntx * B - hc);
    }
    if (STUDENT) {
      // the staging buffer holds the spectrum, so both blocks of rows come to
      // their place in buf now; column 64 of the spectrum goes to a64
      const float2* S1 = a.spec1 + (long long)k * kCol;
      copy_w(buf + blk * 32 * kFP, w, g, i0 - hc, j0 - hc, blk, L);
      stage_slot(st, S1);
      if (L.warp == 0)
        for (int e = threadIdx.x; e < kFT; e += 32) a64[e] = __ldg(S1 + kSlots + e);
      w_rows<true>(nullptr, w, g, i0 - hc, j0 - hc, buf, tw, L, scale);
    } else {
      w_rows<false>(stage, w, g, i0 - hc, j0 - hc, buf, tw, L);
      if (k + 1 < k1)
        copy_w(stage + blk * 32 * kFP, w + g.plane, g, i0 - hc, j0 - hc, blk, L);
    }
    const float2* S = a.spec + (long long)k * kPairSpec + slot_off();
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      float2 kv[STUDENT ? 1 : 16];  // in flight during the transform
      if (!STUDENT) {
#pragma unroll
        for (int i = 0; i < 16; ++i) kv[STUDENT ? 0 : i] = __ldg(S + h * kSlots + 32 * i);
      }
      float2 v[16];
      float2* col = buf + (h == 0 ? m : m2);
      load_col(col, v, L.t, h == 1 && m != 0);
      fft_col(v, col, tw, L.t);
      if (STUDENT) {
        const bool c64 = h == 1 && m == 0;
        const float2* sp = c64 ? a64 + L.t : st + (threadIdx.x & 31);
        const int step = c64 ? 8 : 32;
        if (h == 0) {
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[i] = cfmac(acc[i], v[i], sp[step * i]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            acc2[STUDENT ? i : 0] = cfmac(acc2[STUDENT ? i : 0], v[i], sp[step * i]);
        }
      } else if (h == 1 && m == 0) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          float2* o = a64 + 8 * i + L.t;
          *o = cfmac(*o, v[i], kv[STUDENT ? 0 : i]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] = cfmac(acc[i], v[i], kv[STUDENT ? 0 : i]);
      }
    }
    __syncthreads();  // the buffer is free for the next source
  }
  if (grp >= 0 && a.groups > 1) {
    float2* mine = a.partials + ((long long)tile * a.groups + grp) * kPer;
    store_slot(mine, acc);
    if (STUDENT) {
#pragma unroll
      for (int i = 0; i < 16; ++i) mine[kSlots + slot_off() + 32 * i] = acc2[STUDENT ? i : 0];
    } else {
      for (int e = threadIdx.x; e < kFT; e += blockDim.x) mine[kSlots + e] = a64[e];
    }
    if (!last_group(a, tile)) return;
    const float2* base = a.partials + (long long)tile * a.groups * kPer;
    for (int k = 0; k < a.groups; ++k) {
      const float2* p = base + (long long)k * kPer;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float2 v = __ldcg(p + slot_off() + 32 * i);
        acc[i] = k ? cadd(acc[i], v) : v;
        if (STUDENT) {
          const float2 v2 = __ldcg(p + kSlots + slot_off() + 32 * i);
          acc2[STUDENT ? i : 0] = k ? cadd(acc2[STUDENT ? i : 0], v2) : v2;
        }
      }
      if (!STUDENT)
        for (int e = threadIdx.x; e < kFT; e += blockDim.x) {
          const float2 v = __ldcg(p + kSlots + e);
          a64[e] = k ? cadd(a64[e], v) : v;
        }
    }
    __syncthreads();
  }
  if constexpr (STUDENT) {
    columns_student(acc, acc2, buf, tw, L);
  } else {
    if (!last) {
      publish_part(a, tile, acc, a64, part);
      __syncthreads();
      return;
    }
    columns_gauss(acc, a64, buf, tw, L);
  }
  rows_update<STUDENT>(s, a, 0, i0, j0, buf, tw, L, 1.f / scale);
}

// The same for r > 1, with the accumulators in this item's scratch (`mine`).
// Layout per phase: Gaussian kCol (slots, column 64), Student-t 2 kSlots (the columns m,
// then the partners).
template <bool STUDENT>
__device__ void fft_adjoint_tile_scratch(const Shape& s, const FftLaunch& a, int ty, int tx,
                                         int tile, float2* mine, float2* buf, float2* a64,
                                         const float4* tw, int q0, int q1) {
  const Geom& g = s.g;
  const Lane L;
  const int hc = s.hc, B = kFT - 2 * hc, R2 = s.R2;
  const int i0 = ty * B, j0 = tx * B;
  const int m = L.slot(), m2 = second_col(m);
  const int per = STUDENT ? 2 * kSlots : kCol;
  const int k0 = STUDENT ? 2 * q0 : q0, k1 = STUDENT ? min(2 * q1, s.n) : q1;
  const float scale = STUDENT ? student_scale(a, g, s.n, i0 - hc, j0 - hc) : 1.f;
  float2* stage = buf + kFBuf;
  copy_w(stage + (L.warp >> 3) * 32 * kFP, a.w + (long long)k0 * g.plane, g, i0 - hc, j0 - hc,
         L.warp >> 3, L);
  for (int k = k0; k < k1; ++k) {
    const float2* w = a.w + (long long)k * g.plane;
    if (k + 1 < k1) prefetch_region(w + g.plane, 8, g, i0 - hc, j0 - hc);
    w_rows<STUDENT>(stage, w, g, i0 - hc, j0 - hc, buf, tw, L, scale);
    if (k + 1 < k1)
      copy_w(stage + (L.warp >> 3) * 32 * kFP, w + g.plane, g, i0 - hc, j0 - hc, L.warp >> 3, L);
    float2 f[16], c[16];  // the transforms of column m and of its partner
    load_col(buf + m, f, L.t, false);
    fft_col(f, buf + m, tw, L.t);
    load_col(buf + m2, c, L.t, m != 0);
    fft_col(c, buf + m2, tw, L.t);
    for (int ph = 0; ph < R2; ++ph) {
      float2* o = mine + (long long)ph * per + slot_off();
      if (STUDENT) {
        const float2* S1 = a.spec1 + ((long long)k * R2 + ph) * kCol;
        const float2* sp = S1 + slot_off();
        const float2* sc = m ? sp : S1 + kSlots + L.t;
        const int cstep = m ? 32 : 8;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float2 z = make_float2(0.f, 0.f);
          const float2 of = k > k0 ? o[32 * i] : z, oc = k > k0 ? o[kSlots + 32 * i] : z;
          o[32 * i] = cfmac(of, f[i], sp[32 * i]);
          o[kSlots + 32 * i] = cfmac(oc, c[i], sc[cstep * i]);
        }
      } else {
        const float2* sp = a.spec + ((long long)k * R2 + ph) * kPairSpec + slot_off();
        float2* o64 = mine + (long long)ph * per + kSlots + L.t;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float2 z = make_float2(0.f, 0.f);
          float2 of = k > k0 ? o[32 * i] : z;
          of = cfmac(of, f[i], sp[32 * i]);
          if (m) {
            of = cfmac(of, c[i], sp[kSlots + 32 * i]);
          } else {
            const float2 oc = k > k0 ? o64[8 * i] : z;
            o64[8 * i] = cfmac(oc, c[i], sp[kSlots + 32 * i]);
          }
          o[32 * i] = of;
        }
      }
    }
    __syncthreads();  // the buffer is free for the next source
  }
  const long long gstep = (long long)R2 * per;  // scratch of one group
  int groups = 1;
  if (a.groups > 1) {
    if (!last_group(a, tile)) return;
    groups = a.groups;
    mine = a.scratch + (long long)tile * groups * gstep;
  }
  for (int ph = 0; ph < R2; ++ph) {
    const float2* p = mine + (long long)ph * per;
    float2 f[16], c[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) f[i] = c[i] = make_float2(0.f, 0.f);
    for (int k = 0; k < groups; ++k) {
      const float2* pk = p + k * gstep;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float2 v = __ldcg(pk + slot_off() + 32 * i);
        f[i] = k ? cadd(f[i], v) : v;
        if (STUDENT) {
          const float2 w = __ldcg(pk + kSlots + slot_off() + 32 * i);
          c[i] = k ? cadd(c[i], w) : w;
        }
      }
      if (!STUDENT)
        for (int e = threadIdx.x; e < kFT; e += blockDim.x) {
          const float2 v = __ldcg(pk + kSlots + e);
          a64[e] = k ? cadd(a64[e], v) : v;
        }
    }
    __syncthreads();
    if (STUDENT)
      columns_student(f, c, buf, tw, L);
    else
      columns_gauss(f, a64, buf, tw, L);
    rows_update<STUDENT>(s, a, ph, i0, j0, buf, tw, L, 1.f / scale);
  }
}

// The same for r = 2, Gaussian, with the accumulators in tensor memory (tm) and,
// for column 64, in a64 (four phases); `mine` takes them only where the tile
// has several groups. The terms are added in the other form's order.
__device__ void fft_adjoint_tile_tmem(const Shape& s, const FftLaunch& a, int ty, int tx, int tile,
                                      float2* mine, float2* buf, float2* a64, const float4* tw,
                                      int q0, int q1, uint32_t tm) {
  const Geom& g = s.g;
  const Lane L;
  const int hc = s.hc, B = kFT - 2 * hc;
  const int i0 = ty * B, j0 = tx * B;
  const int m = L.slot(), m2 = second_col(m);
  float2* stage = buf + kFBuf + (L.warp >> 3) * 32 * kFP;
  copy_w(stage, a.w + (long long)q0 * g.plane, g, i0 - hc, j0 - hc, L.warp >> 3, L);
  for (int q = q0; q < q1; ++q) {
    const float2* w = a.w + (long long)q * g.plane;
    if (q + 1 < q1) prefetch_region(w + g.plane, 8, g, i0 - hc, j0 - hc);
    w_rows<false>(buf + kFBuf, w, g, i0 - hc, j0 - hc, buf, tw, L);
    if (q + 1 < q1) copy_w(stage, w + g.plane, g, i0 - hc, j0 - hc, L.warp >> 3, L);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const float2* sp =
          a.spec + (long long)q * kTmPhases * kPairSpec + h * kSlots + slot_off();
      float2 kv[16], v[16];  // phase 0's S in flight during the transform
#pragma unroll
      for (int i = 0; i < 16; ++i) kv[i] = __ldg(sp + 32 * i);
      load_col(buf + (h ? m2 : m), v, L.t, h && m != 0);
      fft_col(v, buf + (h ? m2 : m), tw, L.t);
#pragma unroll 1
      for (int ph = 0; ph < kTmPhases; ++ph) {
        float2 acc[16];
        if (q > q0 || h) {
          tmem_load(acc, tm + 32 * ph);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[i] = make_float2(0.f, 0.f);
        }
        if (h && m == 0) {
          float2* o = a64 + ph * kFT + L.t;
#pragma unroll
          for (int i = 0; i < 16; ++i)
            o[8 * i] = cfmac(q > q0 ? o[8 * i] : make_float2(0.f, 0.f), v[i], kv[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[i] = cfmac(acc[i], v[i], kv[i]);
        }
        if (ph + 1 < kTmPhases) {
          sp += kPairSpec;
#pragma unroll
          for (int i = 0; i < 16; ++i) kv[i] = __ldg(sp + 32 * i);
        }
        __syncwarp();
        tmem_store(tm + 32 * ph, acc);
      }
    }
    __syncthreads();  // the buffer is free for the next source
  }
  const bool groups = a.groups > 1;
  if (groups) {
    for (int ph = 0; ph < kTmPhases; ++ph) {
      float2 acc[16];
      tmem_load(acc, tm + 32 * ph);
      store_slot(mine + (long long)ph * kCol, acc);
      for (int e = threadIdx.x; e < kFT; e += kFThreads)
        mine[(long long)ph * kCol + kSlots + e] = a64[ph * kFT + e];
    }
    if (!last_group(a, tile)) return;
  }
#pragma unroll 1
  for (int ph = 0; ph < kTmPhases; ++ph) {
    float2 acc[16];
    if (!groups) {
      tmem_load(acc, tm + 32 * ph);
    } else {
      const float2* p = a.scratch + ((long long)tile * a.groups * kTmPhases + ph) * kCol;
      for (int k = 0; k < a.groups; ++k, p += (long long)kTmPhases * kCol) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float2 t = __ldcg(p + slot_off() + 32 * i);
          acc[i] = k ? cadd(acc[i], t) : t;
        }
        for (int e = threadIdx.x; e < kFT; e += kFThreads) {
          const float2 t = __ldcg(p + kSlots + e);
          a64[ph * kFT + e] = k ? cadd(a64[ph * kFT + e], t) : t;
        }
      }
      __syncthreads();
    }
    columns_gauss(acc, a64 + ph * kFT, buf, tw, L);
    rows_update<false>(s, a, ph, i0, j0, buf, tw, L);
  }
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------

// pairs [*q0, *q1) of group grp of G over the NP pairs
__device__ __forceinline__ void group_range(int n, int G, int grp, int* q0, int* q1) {
  const int NP = (n + 1) / 2;
  *q0 = (int)((long long)NP * grp / G);
  *q1 = (int)((long long)NP * (grp + 1) / G);
}

// float2 of scratch per (tile, group): x^ of the phases (r > 1), then the
// accumulators
__host__ __device__ inline long long scratch_floats2(int R2, bool student) {
  const long long acc = (long long)R2 * (student ? 2 * kSlots : kCol);
  const long long x = R2 > 1 ? (long long)R2 * kCol : 0;
  return acc > x ? acc : x;
}

// item = tile * groups + group
template <bool R1, bool STUDENT>
__device__ __forceinline__ void forward_item(const Shape& s, const FftLaunch& a, int gxt, int item,
                                             float2* fsm, float2* x64, const float4* tw) {
  const int tile = item / a.groups, grp = item - tile * a.groups;
  int q0, q1;
  group_range(s.n, a.groups, grp, &q0, &q1);
  fft_forward_tile<R1, STUDENT>(s, a, tile / gxt, tile % gxt,
                                R1 ? nullptr : a.scratch + item * scratch_floats2(s.R2, STUDENT),
                                fsm, x64, tw, q0, q1);
}

template <bool R1, bool STUDENT>
__device__ __forceinline__ void adjoint_item(const Shape& s, const FftLaunch& a, int gxt, int item,
                                             float2* fsm, float2* a64, const float4* tw) {
  const int tile = item / a.groups, grp = item - tile * a.groups;
  int q0, q1;
  group_range(s.n, a.groups, grp, &q0, &q1);
  if (R1)
    fft_adjoint_tile<STUDENT>(s, a, tile / gxt, tile % gxt, tile, fsm, a64, tw, q0, q1, grp);
  else
    fft_adjoint_tile_scratch<STUDENT>(
        s, a, tile / gxt, tile % gxt, tile,
        a.scratch + item * (long long)s.R2 * (STUDENT ? 2 * kSlots : kCol), fsm, a64, tw, q0, q1);
}

template <bool R1, bool STUDENT>
__global__ void __launch_bounds__(kFThreads, 1)
    fft_forward_kernel(const Shape s, const FftLaunch a, int gxt) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 x64[kFT];
  init_twiddles(tw);
  after_previous_launch();
  forward_item<R1, STUDENT>(s, a, gxt, blockIdx.x, fsm, x64, tw);
}

template <bool R1, bool STUDENT>
__global__ void __launch_bounds__(kFThreads, 1)
    fft_adjoint_kernel(const Shape s, const FftLaunch a, int gxt) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 a64[kFT];
  init_twiddles(tw);
  after_previous_launch();
  adjoint_item<R1, STUDENT>(s, a, gxt, blockIdx.x, fsm, a64, tw);
}

// r = 2: item = tile * groups + group, x^ (the Gaussian accumulators) in tensor
// memory. 33 x 2048^2 exposures, 85 x 85 PSFs: 4.66 ms an iteration through the
// scratch, 2.40 ms here; 9 x 300 x 280, K = 43: 136 us.
template <bool STUDENT>
__global__ void __launch_bounds__(kFThreads, 1)
    fft_forward_r2_kernel(const Shape s, const FftLaunch a, int gxt) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 x64[kTmPhases * kFT];
  __shared__ uint32_t base;
  init_twiddles(tw);
  after_previous_launch();
  const uint32_t tm = tmem_begin(&base);
  const int tile = blockIdx.x / a.groups;
  int q0, q1;
  group_range(s.n, a.groups, blockIdx.x - tile * a.groups, &q0, &q1);
  fft_forward_tile<false, STUDENT, true>(s, a, tile / gxt, tile % gxt, nullptr, fsm, x64, tw, q0,
                                         q1, -1, 0, tm);
  tmem_end(base);
}

__global__ void __launch_bounds__(kFThreads, 1)
    fft_adjoint_r2_kernel(const Shape s, const FftLaunch a, int gxt) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 a64[kTmPhases * kFT];
  __shared__ uint32_t base;
  init_twiddles(tw);
  after_previous_launch();
  const uint32_t tm = tmem_begin(&base);
  const int tile = blockIdx.x / a.groups;
  int q0, q1;
  group_range(s.n, a.groups, blockIdx.x - tile * a.groups, &q0, &q1);
  fft_adjoint_tile_tmem(s, a, tile / gxt, tile % gxt, tile,
                        a.scratch + (long long)blockIdx.x * kTmPhases * kCol, fsm, a64, tw, q0, q1,
                        tm);
  tmem_end(base);
}

// Equal ranges: CTA b of P takes the units [b U / P, (b+1) U / P) of U.
__device__ __forceinline__ long long split_start(long long U, int P, int b) {
  return (long long)b * U / P;
}

// Split forms (r = 1 Gaussian, at least as many tiles as CTAs): P =
// a.split_ctas persistent CTAs. The Wf = tiles / P whole waves run as one
// CTA per tile would (CTA b takes the tiles b + P i, neighbours side by
// side, so their overlapping regions share the L2); the R = tiles - Wf P
// tiles of the last, partial wave are spread so that no SM idles through it.
// Forward: the (tile, pair) units of the last wave in equal ranges over all
// CTAs (tile-major; a CTA recomputes x^ for each tile it touches).
__global__ void __launch_bounds__(kFThreads, 1)
    fft_forward_split_kernel(const Shape s, const FftLaunch a, int gxt, int tiles) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 x64[kFT];
  init_twiddles(tw);
  after_previous_launch();
  const int P = a.split_ctas, n = (s.n + 1) / 2, b = blockIdx.x;
  const int Wf = tiles / P, R = tiles - Wf * P;
  const long long U = (long long)R * n, base = (long long)Wf * P * n;
  const long long u_end = split_start(U, P, b + 1);
  long long u = split_start(U, P, b);
  for (int i = 0; i < Wf || u < u_end; ++i) {
    int tile, q0 = 0, q1 = n;
    if (i < Wf) {
      tile = b + P * i;
    } else {
      tile = (int)((base + u) / n), q0 = (int)((base + u) % n);
      q1 = (int)min((long long)n, q0 + (u_end - u));
      u += q1 - q0;
    }
    const int next = i + 1 < Wf ? tile + P : -1;
    fft_forward_tile<true, false>(s, a, tile / gxt, tile % gxt, nullptr, fsm, x64, tw, q0, q1,
                                  next >= 0 ? next / gxt : -1, next >= 0 ? next % gxt : 0);
  }
}

// Adjoint: last-wave tile j is cut into k = min(pairs, P / R) parts of
// consecutive pairs, part q on CTA q R + j, which runs it after
// q Wf / (k - 1) of its whole tiles (part 0 first, part k - 1 last), so
// each part finds its predecessor done waves earlier and the last wave
// costs 1 / k of a tile.
__global__ void __launch_bounds__(kFThreads, 1)
    fft_adjoint_split_kernel(const Shape s, const FftLaunch a, int gxt, int tiles) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 a64[kFT];
  init_twiddles(tw);
  after_previous_launch();
  const int P = a.split_ctas, n = (s.n + 1) / 2, b = blockIdx.x;
  const int Wf = tiles / P, R = tiles - Wf * P;
  const int k = R > 0 ? max(1, min(n, P / R)) : 0;
  const int has = b < k * R, q = has ? b / R : 0, j = has ? b % R : 0;
  const int pos = !has ? -1 : (k == 1 ? Wf : q * Wf / (k - 1));  // whole tiles before the part
  for (int it = 0; it < Wf + has; ++it) {
    int tile, k0 = 0, k1 = n, qq = 0, prev = -1;
    bool last = true;
    if (has && it == pos) {
      tile = Wf * P + j, k0 = q * n / k, k1 = (q + 1) * n / k, qq = q;
      prev = q > 0 ? (q - 1) * R + j : -1, last = q == k - 1;
    } else {
      tile = b + P * (it - (has && it > pos));
    }
    const int next = it + 1 < Wf && it != pos ? tile + P : -1;
    fft_adjoint_tile<false>(s, a, tile / gxt, tile % gxt, tile, fsm, a64, tw, k0, k1, -1, qq, prev, last,
                     next >= 0 ? next / gxt : -1, next >= 0 ? next % gxt : 0);
  }
}

// Persistent forms for a batch of FFT jobs: every CTA claims (job, item)
// entries from a device counter until the list is exhausted; jobs whose
// iterations are done are skipped. One launch for the forward passes of all
// jobs, then one for the adjoints (the adjoint reads its neighbours' w).
__device__ __forceinline__ int claim_item(int* counter, int* slot) {
  __syncthreads();  // the previous item's readers of *slot are done
  if (threadIdx.x == 0) *slot = atomicAdd(counter, 1);
  __syncthreads();
  return *slot;
}

__global__ void __launch_bounds__(kFThreads, 1)
    fft_batch_forward_kernel(const FftBatchJob* __restrict__ jobs, const int2* __restrict__ items,
                             const int* __restrict__ n_items, int* __restrict__ counter) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 x64[kFT];
  __shared__ int slot;
  init_twiddles(tw);
  const int total = *n_items;
  for (;;) {
    const int item = claim_item(counter, &slot);
    if (item >= total) break;
    const int2 w = items[item];
    const FftBatchJob& J = jobs[w.x];
    if (J.remaining <= 0) continue;
    if (J.s.R2 == 1)
      forward_item<true, false>(J.s, J.a[J.cur], J.gxt, w.y, fsm, x64, tw);
    else
      forward_item<false, false>(J.s, J.a[J.cur], J.gxt, w.y, fsm, x64, tw);
  }
}

__global__ void __launch_bounds__(kFThreads, 1)
    fft_batch_adjoint_kernel(const FftBatchJob* __restrict__ jobs, const int2* __restrict__ items,
                             const int* __restrict__ n_items, int* __restrict__ counter) {
  extern __shared__ __align__(16) float2 fsm[];
  __shared__ float4 tw[kFT / 2];
  __shared__ float2 a64[kFT];
  __shared__ int slot;
  init_twiddles(tw);
  const int total = *n_items;
  for (;;) {
    const int item = claim_item(counter, &slot);
    if (item >= total) break;
    const int2 w = items[item];
    const FftBatchJob& J = jobs[w.x];
    if (J.remaining <= 0) continue;
    if (J.s.R2 == 1)
      adjoint_item<true, false>(J.s, J.a[J.cur], J.gxt, w.y, fsm, a64, tw);
    else
      adjoint_item<false, false>(J.s, J.a[J.cur], J.gxt, w.y, fsm, a64, tw);
  }
}

__global__ void fft_batch_advance_kernel(FftBatchJob* __restrict__ jobs, int njobs) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < njobs && jobs[j].remaining > 0) {
    jobs[j].remaining -= 1;
    jobs[j].cur ^= 1;
  }
}

// One kernel of an iteration, a programmatic dependent of the launch before where
// both fit on the SMs side by side (200 x 150 x 9, 20 CTAs: 57.1 -> 53.5 us an
// iteration; 143 CTAs: the same; 4096^2 x 33, 152 CTAs: 5.23 -> 5.31 ms). Not
// under stream capture, where the edge would be a programmatic one that
// queries of the graph's dependencies refuse.
template <class Kernel, class... Args>
cudaError_t launch_dependent(Kernel kernel, int grid, cudaStream_t st, Args... args) {
  cudaError_t e = allow_max_dynamic_smem((const void*)kernel);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (e == cudaSuccess) e = cudaStreamIsCapturing(st, &cap);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kFThreads);
  cfg.dynamicSmemBytes = fft_smem_bytes();
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 2 * grid <= kSMs && cap == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <bool R1, bool STUDENT>
cudaError_t launch_pair(const Shape& s, const FftLaunch& a, int gxt, int tiles, cudaStream_t st) {
  const cudaError_t e =
      launch_dependent(fft_forward_kernel<R1, STUDENT>, tiles * a.groups, st, s, a, gxt);
  return e != cudaSuccess
             ? e
             : launch_dependent(fft_adjoint_kernel<R1, STUDENT>, tiles * a.groups, st, s, a, gxt);
}

// r = 2: tensor memory holds the four phases' spectra (not the eight accumulators
// of the heavy-tailed adjoint, nor nine phases)
template <bool STUDENT>
cudaError_t launch_r2(const Shape& s, const FftLaunch& a, int gxt, int tiles, cudaStream_t st) {
  const int grid = tiles * a.groups;
  const cudaError_t e = launch_dependent(fft_forward_r2_kernel<STUDENT>, grid, st, s, a, gxt);
  if (e != cudaSuccess) return e;
  return STUDENT ? launch_dependent(fft_adjoint_kernel<false, true>, grid, st, s, a, gxt)
                 : launch_dependent(fft_adjoint_r2_kernel, grid, st, s, a, gxt);
}

size_t up256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

int fft_tile_side(const Shape& s) { return kFT - 2 * s.hc; }

int fft_tiles_x(const Shape& s) {
  const int B = fft_tile_side(s);
  return (s.g.W + B - 1) / B;
}

int fft_tiles_total(const Shape& s) {
  const int B = fft_tile_side(s);
  return fft_tiles_x(s) * ((s.g.H + B - 1) / B);
}

// Exposure groups per tile: the count that takes the fewest transforms one
// after the other, ceil(tiles G / SMs) rounds of ceil(pairs / G) pairs plus
// about one transform of overhead (x^, or the inverse and the update). It
// depends on the shape alone: a job's bits are the same alone and in a batch.
int fft_groups(const Shape& s) {
  const long long tiles = fft_tiles_total(s);
  const int NP = (s.n + 1) / 2;
  int best = 1;
  long long best_cost = 0;
  for (int G = 1; G <= NP && (G == 1 || tiles * G <= 2 * kSMs); ++G) {
    const long long cost = (tiles * G + kSMs - 1) / kSMs * ((NP + G - 1) / G + 1);
    if (G == 1 || cost < best_cost) {
      best = G;
      best_cost = cost;
    }
  }
  return best;
}

// pair spectra, single spectra (Student-t), scales, w planes, scratch, partials, counters
FftLayout fft_layout(const Shape& s, bool student, int split_ctas) {
  FftLayout L{};
  const size_t NP = (s.n + 1) / 2, tiles = fft_tiles_total(s), G = fft_groups(s);
  const size_t wplanes = student ? s.n : NP;  // float2 planes
  size_t off = 0;
  auto take = [&](size_t bytes) { const size_t o = off; off += up256(bytes); return o; };
  L.spec = take(NP * s.R2 * kPairSpec * sizeof(float2));
  L.spec1 = take(student ? (size_t)s.n * s.R2 * kCol * sizeof(float2) : 0);
  L.scale = take((size_t)(s.n + 1) * sizeof(float));
  L.w = take(wplanes * s.g.plane * sizeof(float2));
  const bool r1 = s.R2 == 1;
  L.scratch = take(r1 ? 0 : tiles * G * scratch_floats2(s.R2, student) * sizeof(float2));
  // slots of the split launch (one per CTA) and of the groups, which a shape of the
  // split launch has in a batch where the device has few SMs
  const bool split = r1 && !student && split_ctas > 0 && tiles >= (size_t)split_ctas;
  const size_t slots = std::max(split ? (size_t)split_ctas : 0, r1 && G > 1 ? tiles * G : 0);
  L.partials = take(slots * (student ? 2 * kSlots : kCol) * sizeof(float2));
  L.counters = take(split || G > 1 ? tiles * sizeof(int) : 0);
  L.total = off;
  return L;
}

// the transform buffer and the staging buffer (the forward pass: 4 KB of
// spectrum per warp; the adjoint: 64 rows of the next w region)
size_t fft_smem_bytes() {
  return (size_t)(kFBuf + std::max(kFThreads / 32 * kStage, 64 * kFP)) * sizeof(float2);
}

cudaError_t launch_fft_spectra(const Shape& s, const float* ka, float* inv_scale, float2* spec,
                               float2* spec1, cudaStream_t st) {
  const size_t smem = fft_smem_bytes();
  cudaError_t e = allow_max_dynamic_smem((const void*)fft_spectra_kernel);
  if (e != cudaSuccess) return e;
  fft_scale_kernel<<<s.n, 256, 0, st>>>(ka, s.Kc * s.KP, s.R2, inv_scale);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  fft_scaled_kernel<<<1, 256, 0, st>>>(s.n, inv_scale);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  fft_spectra_kernel<<<(s.n + 1) / 2 * s.R2, kFThreads, smem, st>>>(ka, inv_scale, s.n, s.R2, s.Kc,
                                                                    s.KP, false, spec);
  if ((e = cudaGetLastError()) != cudaSuccess || !spec1) return e;
  fft_spectra_kernel<<<s.n * s.R2, kFThreads, smem, st>>>(ka, inv_scale, s.n, s.R2, s.Kc, s.KP,
                                                          true, spec1);
  return cudaGetLastError();
}

cudaError_t launch_fft_batch(const FftBatchJob* jobs, int njobs, const int2* items,
                             const int* n_items, int* counters, int ctas, cudaStream_t st) {
  const size_t smem = fft_smem_bytes();
  cudaError_t e = allow_max_dynamic_smem((const void*)fft_batch_forward_kernel);
  if (e == cudaSuccess) e = allow_max_dynamic_smem((const void*)fft_batch_adjoint_kernel);
  if (e == cudaSuccess) e = cudaMemsetAsync(counters, 0, 2 * sizeof(int), st);
  if (e != cudaSuccess) return e;
  fft_batch_forward_kernel<<<ctas, kFThreads, smem, st>>>(jobs, items, n_items, counters);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  fft_batch_adjoint_kernel<<<ctas, kFThreads, smem, st>>>(jobs, items, n_items, counters + 1);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  fft_batch_advance_kernel<<<(njobs + 127) / 128, 128, 0, st>>>(const_cast<FftBatchJob*>(jobs),
                                                                njobs);
  return cudaGetLastError();
}

cudaError_t launch_fft_iter(const Shape& s, const FftLaunch& a, cudaStream_t st) {
  const int gxt = fft_tiles_x(s), tiles = fft_tiles_total(s);
  if (s.R2 == kTmPhases)
    return a.nu > 0.f ? launch_r2<true>(s, a, gxt, tiles, st)
                      : launch_r2<false>(s, a, gxt, tiles, st);
  if (a.nu > 0.f)
    return s.R2 == 1 ? launch_pair<true, true>(s, a, gxt, tiles, st)
                     : launch_pair<false, true>(s, a, gxt, tiles, st);
  if (s.R2 > 1) return launch_pair<false, false>(s, a, gxt, tiles, st);
  if (a.split_ctas <= 0 || tiles < a.split_ctas)
    return launch_pair<true, false>(s, a, gxt, tiles, st);
  const cudaError_t e =
      launch_dependent(fft_forward_split_kernel, a.split_ctas, st, s, a, gxt, tiles);
  return e != cudaSuccess
             ? e
             : launch_dependent(fft_adjoint_split_kernel, a.split_ctas, st, s, a, gxt, tiles);
}

}  // namespace emd
