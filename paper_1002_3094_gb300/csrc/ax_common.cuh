// Small device helpers: vector loads, warp/CTA reductions in FP64.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstdint>
#include "ax_internal.cuh"

namespace ax {

template <typename T> struct VecT;
template <> struct VecT<float> { using type = float4; static constexpr int n = 4; };
template <> struct VecT<double> { using type = double2; static constexpr int n = 2; };

template <typename T>
__device__ __forceinline__ void load_vec(const T *p, T (&v)[VecT<T>::n]);
template <>
__device__ __forceinline__ void load_vec<float>(const float *p, float (&v)[4]) {
  float4 t = *reinterpret_cast<const float4 *>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <>
__device__ __forceinline__ void load_vec<double>(const double *p, double (&v)[2]) {
  double2 t = *reinterpret_cast<const double2 *>(p);
  v[0] = t.x; v[1] = t.y;
}
template <typename T>
__device__ __forceinline__ void store_vec(T *p, const T (&v)[VecT<T>::n]);
template <>
__device__ __forceinline__ void store_vec<float>(float *p, const float (&v)[4]) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ void store_vec<double>(double *p, const double (&v)[2]) {
  *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Deterministic CTA sum (fixed order); result valid in thread 0.
// `red` must hold blockDim.x / 32 doubles.
__device__ __forceinline__ double block_sum(double v, double *red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int w = 0; w < nw; ++w) s += red[w];
  }
  return s;
}

// Sum of N FP32 values of every lane of a warp, returned in FP64.  GB300 adds two FP64
// numbers per clock and SM, so an FP64 shuffle tree holds that pipe for 80 cycles a
// warp.  Here the values are cut to integers of 60 bits below the largest one's exponent
// (three words of 20 bits with room for the sums) and added exactly by the warp's
// integer reductions: what is lost is at most 32 N 2^-60 of the largest value and the
// rounding of the result, less than an FP64 tree loses (5 2^-53 of the sum of
// magnitudes for N = 1), and no sum overflows.  Values that are not finite are summed in
// FP64.
template <int N>
__device__ __forceinline__ double warp_sum_fp32(const float (&v)[N]) {
  unsigned top = 1;
#pragma unroll
  for (int i = 0; i < N; ++i) top = max(top, (__float_as_uint(v[i]) >> 23) & 255u);
  top = __reduce_max_sync(0xffffffffu, top);
  if (top == 255u) {
    double d = 0.0;
    for (int i = 0; i < N; ++i) d += (double)v[i];
    return warp_sum(d);
  }
  int w0 = 0, w1 = 0, w2 = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const unsigned b = __float_as_uint(v[i]), f = (b >> 23) & 255u;
    const unsigned mant = (b & 0x7FFFFFu) | (f != 0 ? 0x800000u : 0u);
    const unsigned long long X = ((unsigned long long)mant << 36) >> min(top - max(f, 1u), 63u);
    const int sgn = (int)b >> 31;  // 0 or -1
    w0 += ((int)(X >> 40) ^ sgn) - sgn;
    w1 += ((int)(X >> 20 & 0xFFFFF) ^ sgn) - sgn;
    w2 += ((int)(X & 0xFFFFF) ^ sgn) - sgn;
  }
  w0 = __reduce_add_sync(0xffffffffu, w0);
  w1 = __reduce_add_sync(0xffffffffu, w1);
  w2 = __reduce_add_sync(0xffffffffu, w2);
  // sum 2^-5 in units of 2^(top - 127 - 23 - 36) as one integer of at most 63 bits
  // (N <= 8), rounded to a double by its bits
  const long long S = ((long long)w0 << 35) + ((((long long)w1 << 20) + w2) >> 5);
  if (S == 0) return 0.0;
  const unsigned long long a = (unsigned long long)(S < 0 ? -S : S);
  const int lz = __clzll((long long)a);
  unsigned long long r = a << lz;
  r = (r >> 11) + ((r >> 10) & 1);  // 2^52 .. 2^53
  const unsigned long long bits = ((unsigned long long)(1023 + 63 - lz + 5 + (int)top - 186 - 1) << 52) + r;
  return __longlong_as_double((long long)(bits | (S < 0 ? 1ull << 63 : 0ull)));
}
__device__ __forceinline__ double warp_sum_of(float v) {
  const float w[1] = {v};
  return warp_sum_fp32(w);
}
__device__ __forceinline__ double warp_sum_of(double v) { return warp_sum(v); }

// Sums of many FP32 values as three FP32 numbers, h + m + l: the rounding errors of h
// (two-sum, exact) are summed in m and those of m in l, so that only roundings of l are
// lost.  A sum that leaves FP32's range is infinite, one of values that are not finite
// what their FP32 sum is.
struct Sum3 {
  float h = 0.f, m = 0.f, l = 0.f;
  __device__ __forceinline__ static float two_sum(float a, float b, float &err) {
    const float s = a + b, bb = s - a;
    err = (a - (s - bb)) + (b - bb);
    return s;
  }
  __device__ __forceinline__ void add(float v) {
    float e1, e2;
    h = two_sum(h, v, e1);
    m = two_sum(m, e1, e2);
    l += e2;
  }
  __device__ __forceinline__ void add(const Sum3 &o) {
    float e1, e2, e3;
    h = two_sum(h, o.h, e1);
    m = two_sum(m, o.m, e2);
    m = two_sum(m, e1, e3);
    l = (l + o.l) + (e2 + e3);
  }
  // to words of at most 2^-24 each of the one before (every 256 values: the errors of
  // l then stay below those of FP64 sums)
  __device__ __forceinline__ void renorm() {
    h = two_sum(h, m, m);
    m = two_sum(m, l, l);
  }
  __device__ __forceinline__ float value() const { return isfinite(h) ? h + (m + l) : h; }
};

template <typename T>
__device__ __forceinline__ double block_sum_of(T v, double *red) {
  const double w = warp_sum_of(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = w;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int i = 0; i < nw; ++i) s += red[i];
  }
  return s;
}

__device__ __forceinline__ bool rhs_selected(const RhsState *st, int mask, int m) {
  if (mask == kDue) return st[m].state == kActive && st[m].due != 0;
  if (mask == kLive) return st[m].state == kActive || st[m].state == kRedo;
  return mask < 0 || st[m].state == mask;
}

// ---- mbarrier and bulk-copy primitives (PTX) --------------------------------
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the phase with the given parity (at most `polls` tries);
// false when it expired.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, unsigned polls) {
  for (unsigned i = 0; i < polls; ++i)
    if (mbar_try(bar, parity)) return true;
  return false;
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// ---------------------------------------------------------------------------
// BF16 operand of the tensor-core transform ("split" layout).  A field x is
// stored as x = hi + lo, hi = bf16(x), lo = bf16(x - hi), in tiles of 128 rows
// x 64 positions per right-hand side: tile (m, row / 128, pos / 64) is 32 KB,
// the 16 KB of high parts and then the 16 KB of low parts, each as 8 x 8 core
// matrices of 16-byte rows, element (row, pos) at byte
//   (row % 128 / 8) 1024 + (pos % 64 / 8) 128 + (row % 8) 16 + (pos % 8) 2.
// Columns are stored even ones first (the operand order of the transform's
// even / odd split): column c at position c / 2 if c is even, else at
// kbe 64 + c / 2, with kbe = ceil(n8 / 2 / 64) tiles of even columns and as
// many of odd ones, n8 = n rounded up to 8.  Writers store whole chunks of 8
// columns c < n8 only (chunk starts c < n), which keeps every position inside.
// A tile is copied to shared memory as it is.  Padding rows and positions
// hold zeros (the buffer is zeroed when allocated and never written there).
// ---------------------------------------------------------------------------
constexpr int kSplitTileBytes = 32768;

__device__ __forceinline__ int split_pos(int c, int kbe) { return (c & 1) ? kbe * 64 + (c >> 1) : (c >> 1); }
__device__ __forceinline__ size_t split_byte(int m, int row, int pos, int mtiles, int ktiles) {
  return (((size_t)m * mtiles + (row >> 7)) * ktiles + (pos >> 6)) * (size_t)kSplitTileBytes +
         ((row & 127) >> 3) * 1024 + ((pos & 63) >> 3) * 128 + (row & 7) * 16 + (pos & 7) * 2;
}
__device__ __forceinline__ unsigned bf16_pack2(float a, float b) {
  // round-to-nearest-even BF16 of a (low half, lower address) and b, by the
  // packed conversion instruction
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const unsigned *>(&h);
}
__device__ __forceinline__ float bf16_round(float a) { return __bfloat162float(__float2bfloat16_rn(a)); }
// The two BF16 halves of a packed pair as FP32 (exact).
__device__ __forceinline__ float bf16_lo(unsigned p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf16_hi(unsigned p) { return __uint_as_float(p & 0xFFFF0000u); }
// The same operand stored by modes, for the inverse transform (the tensor core reads
// either): in each 16 KB half of a tile, blocks of 64 rows x 8 positions (1 KB), the
// positions' blocks consecutive, each position a run of 64 rows (128 bytes) whose
// 16-byte pieces are swizzled by the position (the 128-byte swizzle).  Byte of 8
// consecutive rows from `row` on:
__device__ __forceinline__ size_t split_t_byte(int m, int row, int pos, int mtiles, int ktiles) {
  return (((size_t)m * mtiles + (row >> 7)) * ktiles + (pos >> 6)) * (size_t)kSplitTileBytes +
         ((row & 127) >> 6) * 8192 + ((pos & 63) >> 3) * 1024 + (pos & 7) * 128 +
         ((((row & 63) >> 3) ^ (pos & 7)) << 4) + (row & 7) * 2;
}
// Writes the 8 consecutive columns col .. col + 7 (col % 8 == 0) of one row:
// the 4 even ones and the 4 odd ones each as 8 bytes of high and of low parts.
__device__ __forceinline__ void split_store8(unsigned char *split, int m, int row, int col, int mtiles, int ktiles,
                                             int kbe, const float (&x)[8]) {
  unsigned he[2], le[2], ho[2], lo[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    he[e] = bf16_pack2(x[4 * e], x[4 * e + 2]);
    ho[e] = bf16_pack2(x[4 * e + 1], x[4 * e + 3]);
    le[e] = bf16_pack2(x[4 * e] - bf16_lo(he[e]), x[4 * e + 2] - bf16_hi(he[e]));
    lo[e] = bf16_pack2(x[4 * e + 1] - bf16_lo(ho[e]), x[4 * e + 3] - bf16_hi(ho[e]));
  }
  unsigned char *te = split + split_byte(m, row, split_pos(col, kbe), mtiles, ktiles);
  unsigned char *to = split + split_byte(m, row, split_pos(col + 1, kbe), mtiles, ktiles);
  *reinterpret_cast<uint2 *>(te) = make_uint2(he[0], he[1]);
  *reinterpret_cast<uint2 *>(te + kSplitTileBytes / 2) = make_uint2(le[0], le[1]);
  *reinterpret_cast<uint2 *>(to) = make_uint2(ho[0], ho[1]);
  *reinterpret_cast<uint2 *>(to + kSplitTileBytes / 2) = make_uint2(lo[0], lo[1]);
}

// Writes the 4 consecutive columns col .. col + 3 (col % 4 == 0) of one row:
// the 2 even ones and the 2 odd ones each as 4 bytes of high and of low parts.
__device__ __forceinline__ void split_store4(unsigned char *split, int m, int row, int col, int mtiles, int ktiles,
                                             int kbe, const float (&x)[4]) {
  const unsigned he = bf16_pack2(x[0], x[2]), ho = bf16_pack2(x[1], x[3]);
  unsigned char *te = split + split_byte(m, row, split_pos(col, kbe), mtiles, ktiles);
  unsigned char *to = split + split_byte(m, row, split_pos(col + 1, kbe), mtiles, ktiles);
  *reinterpret_cast<unsigned *>(te) = he;
  *reinterpret_cast<unsigned *>(te + kSplitTileBytes / 2) = bf16_pack2(x[0] - bf16_lo(he), x[2] - bf16_hi(he));
  *reinterpret_cast<unsigned *>(to) = ho;
  *reinterpret_cast<unsigned *>(to + kSplitTileBytes / 2) = bf16_pack2(x[1] - bf16_lo(ho), x[3] - bf16_hi(ho));
}

// Folded input of the tensor-core cosine forward transform for the 8
// positions k0 .. k0 + 7 (k0 % 8 == 0) of one row, from x[e] = r_{k0+e} and
// xm[e] = r_{n-1-k0-e}: u_k = r_k + r_{n-1-k} at position k of the first K
// half, w_k = r_k - r_{n-1-k} at position kbe 64 + k of the second, for
// k < ceil(n/2) (the middle entry of odd n: u = r, w = 0), zeros after.
__device__ __forceinline__ void fold_store8(unsigned char *split, int m, int row, int k0, int n, int mtiles,
                                            int ktiles, int kbe, const float (&x)[8], const float (&xm)[8]) {
  const int ne = (n + 1) >> 1;
  unsigned uh[4], ul[4], wh[4], wl[4];
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    float u2[2], w2[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int k = k0 + e + j;
      const bool mid = 2 * k + 1 == n;
      u2[j] = k < ne ? (mid ? x[e + j] : x[e + j] + xm[e + j]) : 0.f;
      w2[j] = (k < ne && !mid) ? x[e + j] - xm[e + j] : 0.f;
    }
    const float uh0 = bf16_round(u2[0]), uh1 = bf16_round(u2[1]);
    const float wh0 = bf16_round(w2[0]), wh1 = bf16_round(w2[1]);
    uh[e / 2] = bf16_pack2(uh0, uh1);
    ul[e / 2] = bf16_pack2(u2[0] - uh0, u2[1] - uh1);
    wh[e / 2] = bf16_pack2(wh0, wh1);
    wl[e / 2] = bf16_pack2(w2[0] - wh0, w2[1] - wh1);
  }
  unsigned char *pu = split + split_byte(m, row, k0, mtiles, ktiles);
  unsigned char *pw = split + split_byte(m, row, kbe * 64 + k0, mtiles, ktiles);
  *reinterpret_cast<uint4 *>(pu) = make_uint4(uh[0], uh[1], uh[2], uh[3]);
  *reinterpret_cast<uint4 *>(pu + kSplitTileBytes / 2) = make_uint4(ul[0], ul[1], ul[2], ul[3]);
  *reinterpret_cast<uint4 *>(pw) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
  *reinterpret_cast<uint4 *>(pw + kSplitTileBytes / 2) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
}

}  // namespace ax
