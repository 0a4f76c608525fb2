// FP64 z-transforms on the tensor cores by exact integer products.
//
// GB300 issues two FP64 operations per clock and SM, so the FP64 FFT of the plain
// method (100-200 operations per point) is bound by that pipe: 1.42 ms for 8192
// rows of 1024, against 0.02 ms for reading and writing them.  The BF16 tensor
// cores are some 1600 times as fast, and exact on small integers: following
// Ozaki, Ogita, Oishi and Rump ("Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012) each row of the input and the
// transform matrix are written as sums of integer matrices with few bits,
//
//     x = 2^(e-55) sum_s X_s 128^(7-s),   S = 2^(eS-54) sum_t S_t 128^(7-t),
//
// s, t = 0..7, |X_s|, |S_t| <= 64 but |X_0| <= 128 (all exact in BF16): 56 bits
// relative to the row's largest entry, e its exponent.  The products with s + t =
// d go to one FP32 accumulator: X_0 S_d and d others, each a sum over at most 512
// positions, together at most 512 64 (128 + 64 d) = (2 + d) 2^21: an integer of at
// most 2^24, so exact, for d <= 6 (for d = 7, should every digit be extreme at
// once, off by one unit of a weight of 2^-62 of the largest product).  The 36
// products with d <= 7 are formed; the rest would change the result by about 2^-56
// of the row's norm.  The 8 accumulators are put together in two 64-bit integers
// and rounded to FP64 once.  A row whose entries are small beside its largest (the sum
// of |X_0| stays below 512 128 with one bit more) gets that bit, |X_0| <= 256: there
// the rounding of the digits, not that of the result, would be the larger error.
// Error against 64-bit significands, in 2^-53 of the row's norm, rows of normal deviates
// and single, wide-ranged, constant, smooth and decaying ones, 11 lengths from 128 to
// 1024, both boundaries: 0.65-0.80 on average over the normal deviates, at most 2.7 (the
// FFT: 1.9-6.8, 7.3).
//
// Even / odd split as in ax_dst_gemm.cu: P = (even input columns) S and Q = (odd
// input columns) S over the first ceil(n/2) output columns, out[l] = P + Q,
// out[n-1-l] = P - Q (cosine forward: folded input, even columns from P, odd from
// Q).  A cluster of two CTAs computes 128 rows x 64 columns (or 32), one P and one Q,
// whose 8 accumulators of 64 columns fill its TMEM; each then sends the other half of
// its sums through distributed shared memory and finishes half of the columns.  (One
// CTA for both, P before Q: 470 us in place of 405 at 8192 x 1024, then, and 1.6 times the
// time where a launch has few tiles.)  K blocks of 32 (64 KB of input digits, 32 KB
// of matrix digits) come by bulk copies through two stages (16 through four: 1.07
// times the time).  What bounds the products at 1024 points, some 90 000 cycles per
// CTA: 1152 MMAs of 50 cycles (6 KB of operands each through shared memory), then
// 16 000 cycles of FP64 pipe in the drain with no MMAs beside it, as the accumulators
// fill TMEM, and the first copies.  Both kernels, 8192 rows of 1024: 392 us against
// the FFT's 1503; 4000 rows of 511: 84 against 190.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>
#include "ax_finish.cuh"

namespace ax {

namespace {

constexpr int kDM = 128, kDN = 64, kDK = 32, kSlices = 8;
constexpr int kDATile = kDM * kDK * 2, kDBTile = kDN * kDK * 2;  // one slice, bytes
constexpr int kDStages = 2;
constexpr int kDEpiWarps = 8;
constexpr int kDThreads = 128 + 32 * kDEpiWarps;
constexpr unsigned kDPolls = 1u << 22;
// Shapes for DN output columns per CTA: a stage, the exchange with the peer CTA
template <int DN>
struct DigitTile {
  static constexpr int btile = DN * kDK * 2, stage = kSlices * (kDATile + btile);
  static constexpr size_t smem = (size_t)kDStages * stage + DN / 2 * kDM * 8 + 1024;
};

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory descriptor: K-major, no swizzle; core matrices of 8 rows x 16
// bytes, 128 bytes apart along K, kDK 16 bytes apart along the rows.
__device__ __forceinline__ uint64_t digit_desc(const void *p) {
  return (uint64_t)((smem_u32(p) >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)((unsigned)kDK * 16u >> 4) << 32) |
         (1ull << 46);
}
template <int DN>
constexpr unsigned kDIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(DN >> 3) << 17) |
                             ((unsigned)(kDM >> 4) << 24);
// USE: 0 the input operand is read and kept in the collector buffer, 1 taken from
// it, 2 taken for the last time.
template <int DN, int USE>
__device__ __forceinline__ void digit_mma(unsigned d, uint64_t a, uint64_t b, unsigned accumulate) {
#define AX_DIGIT_MMA(OP)                                                                    \
  asm volatile(                                                                             \
      "{\n\t.reg .pred p;\n\t"                                                              \
      "setp.ne.b32 p, %4, 0;\n\t"                                                           \
      "tcgen05.mma.cta_group::1.kind::f16.collector::a::" OP " [%0], %1, %2, %3, p;\n\t}" :: \
          "r"(d), "l"(a), "l"(b), "r"(kDIdesc<DN>), "r"(accumulate)                             \
      : "memory")
  if constexpr (USE == 0) AX_DIGIT_MMA("fill");
  else if constexpr (USE == 1) AX_DIGIT_MMA("use");
  else AX_DIGIT_MMA("lastuse");
#undef AX_DIGIT_MMA
}
__device__ __forceinline__ void digit_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// 32 lanes x 8 columns
__device__ __forceinline__ void tmem_ld8(unsigned addr, unsigned (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
}

// The pair of CTAs of a cluster: all threads of both arrive and wait, on every path.
__device__ __forceinline__ void pair_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void pair_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ unsigned peer_addr(const void *p, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"((unsigned)rank));
  return r;
}
__device__ __forceinline__ void peer_store(double *p, double v, int rank) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(peer_addr(p, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ void peer_arrive(uint64_t *bar, int rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(peer_addr(bar, rank)) : "memory");
}
// Waits (at most `polls` tries) for the peer's arrivals of phase 0.
__device__ __forceinline__ bool peer_wait(uint64_t *bar, unsigned polls) {
  for (unsigned i = 0; i < polls; ++i) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar))
        : "memory");
    if (ok) return true;
  }
  return false;
}

// Byte offset of (row, k) in a slice tile of a K block.
__device__ __forceinline__ int digit_byte(int row, int k) {
  return (row >> 3) * (kDK * 16) + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// X (|X| <= 2^57) as 8 digits, most significant first: [-64, 63], the first
// [-256, 256].  With 64 added at each digit but the first, the digits are plain bit
// fields; a field becomes a float by the bits of 2^23 + field (FP32 and integer
// operations: the conversion instructions have an eighth of their rate).
__device__ __forceinline__ void digits_of(long long X, float (&d)[kSlices]) {
  constexpr long long kBias = 64ll * 0x40810204081ll;  // 64 sum of 128^k, k = 0 .. 6
  const unsigned long long Y = (unsigned long long)(X + kBias);
#pragma unroll
  for (int s = kSlices - 1; s > 0; --s) {
    const int at = 7 * (kSlices - 1 - s);
    d[s] = __uint_as_float(((unsigned)(Y >> at) & 127u) | 0x4B000000u) - 8388672.f;
  }
  d[0] = __int_as_float(0x4B400000 + (int)((long long)Y >> 49)) - 12582912.f;
}
// Two floats that BF16 holds exactly, packed.
__device__ __forceinline__ unsigned bf16_pack_exact(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// v 2^(bits - e) rounded to an integer (bits = 54 or 55), for a finite v below
// 2^(e+2), from the bits of v.
__device__ __forceinline__ long long fixed_point(double v, int e, int bits) {
  const long long b = __double_as_longlong(v);
  const int f = (int)((b >> 52) & 0x7FF);
  unsigned long long mant = (unsigned long long)b << 11;  // 1.mantissa at bit 63
  if (f != 0) mant |= 1ull << 63;
  const int r = 62 - bits + (e - ((f != 0 ? f : 1) - 1023));  // one bit kept below the unit
  const unsigned long long t = r < 64 ? mant >> r : 0ull;
  const long long X = (long long)((t + 1) >> 1);
  return b < 0 ? -X : X;
}

// ---------------------------------------------------------------------------
// Input digits: 8 rows per CTA.  A warp per row first forms the row (with update:
// x += alpha p, r -= alpha q and the ||r||^2 partials of PCG) and its largest
// magnitude; then 8 rows x 64 columns per warp are cut into digits, whose 16-byte
// pieces fill whole 128-byte core matrices.  Columns past n and the rest of the
// last K block are written as zeros.  Bound by integer issue (some 45 operations per
// value for the digits) and, with update, the latency of the row pass: 63 us for 8192
// rows of 1024 (30 at the copy rate).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 4) digit_split_kernel(const DigitArgs a) {
  __shared__ double red[8];
  __shared__ int s_e[8];
  const int m = blockIdx.y;
  if (!rhs_selected(a.st, a.mask, m)) return;
  const int n = a.n, row0 = blockIdx.x * 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t base = (size_t)m * (size_t)a.in_field;
  const double *src = a.r != nullptr ? a.r : a.in;
  // 16-byte loads (a caller's rows may start at any element)
  const bool pairs = (a.in_pitch & 1) == 0 && (a.in_field & 1) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  double acc = 0.0;
  {
    const int row = row0 + warp;
    // the largest magnitude (as bits) and an upper bound of the magnitudes' sum:
    // FP32 numbers cut from the FP64 bits, one unit up (0 below 2^-126)
    unsigned long long top = 0;
    float total = 0.f;
    auto see = [&](double v) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
      top = max(top, b);
      const int ex = (int)(b >> 52) - 1023 + 127;
      total += ex <= 0 ? 0.f : ex >= 254 ? INFINITY : __int_as_float((ex << 23 | (int)(b >> 29 & 0x7FFFFF)) + 1);
    };
    if (row < a.rows) {
      const size_t rb = base + (size_t)row * a.in_pitch;
      if (a.r != nullptr) {
        const double alpha = a.st[m].alpha;
        const double *p = (a.st[m].iters & 1) ? a.pa : a.pb;
        #pragma unroll 2
        for (int k = lane * 2; k < n; k += 64) {
          double2 rv = *reinterpret_cast<const double2 *>(a.r + rb + k);
          const double2 qv = *reinterpret_cast<const double2 *>(a.in + rb + k);
          double2 xv = *reinterpret_cast<const double2 *>(a.x + rb + k);
          const double2 pv = *reinterpret_cast<const double2 *>(p + rb + k);
          xv.x = fma(alpha, pv.x, xv.x);
          xv.y = fma(alpha, pv.y, xv.y);
          rv.x = fma(-alpha, qv.x, rv.x);
          rv.y = fma(-alpha, qv.y, rv.y);
          acc = fma(rv.x, rv.x, acc);
          acc = fma(rv.y, rv.y, acc);
          *reinterpret_cast<double2 *>(a.x + rb + k) = xv;
          *reinterpret_cast<double2 *>(a.r + rb + k) = rv;
          see(rv.x);
          see(rv.y);  // (zero in the padding column of odd n)
        }
      } else {
#pragma unroll 4
        for (int k = lane; k < n; k += 32) see(src[rb + k]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
      total += __shfl_xor_sync(0xffffffffu, total, o);
    }
    const int f = (int)(top >> 52);
    // exponent of the largest entry; a folded input can be twice as large
    int e = (f != 0 ? f : 1) - 1023 + (a.fold ? 1 : 0);
    // one bit more where the sum over the row of |v| 2^(7-e) + 1, a bound of the
    // first digits' sum of either half, folded or not, stays below 512 128
    if (e > -100 && e < 100 && total * __int_as_float((7 - e + 127) << 23) * 1.0001f + (float)n <= 65536.f) e -= 1;
    if (lane == 0) {
      s_e[warp] = f == 0x7FF ? 1 << 20 : e;
      // the row's exponent for the products (NaN for a row that is not finite)
      if (row < a.rows) a.scale[(size_t)m * a.mtiles * kDM + row] = f == 0x7FF ? __longlong_as_double(0x7FF8000000000000ll) : (double)e;
    }
  }
  __syncthreads();
  const int ne = (n + 1) >> 1, kbh = (ne + kDK - 1) / kDK;  // K blocks per half
  const int r = lane >> 2, row = row0 + r, e = s_e[r];
  // a folded sum of entries from 2^1023 on can exceed the FP64 range: halves are folded
  const bool halves = a.fold && e > 1023;
  const int ef = halves ? e - 1 : e;
  const size_t rb = base + (size_t)row * a.in_pitch;
  const bool row_ok = row < a.rows && e < (1 << 20);
  // a task: 8 positions of both halves (16 columns)
  for (int g = warp * 4 + (lane & 3); g < kbh * (kDK / 8); g += 32) {
    double v[2][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = g * 8 + i;
      v[0][i] = v[1][i] = 0.0;
      if (!row_ok) continue;
      if (!a.fold) {
        if (!pairs) {
          if (2 * k < n) v[0][i] = src[rb + 2 * k];
          if (2 * k + 1 < n) v[1][i] = src[rb + 2 * k + 1];
        } else if (2 * k < n) {  // an even pitch: the pair lies in the row
          const double2 t = *reinterpret_cast<const double2 *>(src + rb + 2 * k);
          v[0][i] = t.x;
          if (2 * k + 1 < n) v[1][i] = t.y;
        }
      } else if (k < ne) {  // u_k = r_k + r_{n-1-k}, w_k = r_k - r_{n-1-k} (the middle entry of odd n once)
        double x = src[rb + k], y = src[rb + n - 1 - k];
        if (halves) {
          x *= 0.5;
          y *= 0.5;
        }
        const bool mid = 2 * k + 1 == n;
        v[0][i] = mid ? x : x + y;
        v[1][i] = mid ? 0.0 : x - y;
      }
    }
    const int kb = g / (kDK / 8);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      unsigned pk[kSlices][4];
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        float d0[kSlices], d1[kSlices];
        digits_of(fixed_point(v[h][i], ef, 55), d0);
        digits_of(fixed_point(v[h][i + 1], ef, 55), d1);
#pragma unroll
        for (int s = 0; s < kSlices; ++s) pk[s][i >> 1] = bf16_pack_exact(d0[s], d1[s]);
      }
      unsigned char *t = a.digits + (((size_t)m * a.mtiles + (row >> 7)) * 2 * kbh + h * kbh + kb) * (size_t)(kSlices * kDATile) +
                         digit_byte(row & 127, g % (kDK / 8) * 8);
#pragma unroll
      for (int s = 0; s < kSlices; ++s)
        *reinterpret_cast<uint4 *>(t + s * kDATile) = make_uint4(pk[s][0], pk[s][1], pk[s][2], pk[s][3]);
    }
  }
  if (a.partial != nullptr) {
    const double sum = block_sum(acc, red);
    if (threadIdx.x == 0) a.partial[(size_t)m * kPartialStride + blockIdx.x] = sum;
    finish_rhs(a.fin, m, gridDim.x, a.partial + (size_t)m * kPartialStride, (int)gridDim.x, red);
  }
}

// hi 2^28 + lo rounded once, |hi|, |lo| < 2^50, in two FP64 operations: the bits of
// 1.5 2^80 plus hi are those of 1.5 2^80 + hi 2^28, and the bits of 1.5 2^52 plus lo
// those of 1.5 2^52 + lo; the difference with the constants' sum is exact.
__device__ __forceinline__ double join(long long hi, long long lo) {
  const double h = __longlong_as_double(0x44F8000000000000ll + hi), l = __longlong_as_double(0x4338000000000000ll + lo);
  return (h - 0x1.8000001800000p+80) + l;
}
// v 2^sh in integer operations where v and the result are normal numbers
__device__ __forceinline__ double scaled(double v, int sh) {
  const int ex = (__double2hiint(v) >> 20) & 0x7FF;
  if (ex >= 1 && ex + sh >= 1 && ex + sh <= 2046 && sh < 4096)
    return __hiloint2double(__double2hiint(v) + sh * (1 << 20), __double2loint(v));
  return sh >= 4096 ? __longlong_as_double(0x7FF8000000000000ll) : ldexp(v, sh);
}

// ---------------------------------------------------------------------------
// The products.
// ---------------------------------------------------------------------------
template <int DN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kDThreads, 1) digit_gemm_kernel(const DigitArgs a) {
  using T = DigitTile<DN>;
  extern __shared__ __align__(1024) unsigned char dsm_raw[];
  unsigned char *dsm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(dsm_raw) + 1023) & ~uintptr_t(1023));
  double *xch = reinterpret_cast<double *>(dsm + kDStages * T::stage);  // [column][row] from the peer
  __shared__ __align__(8) uint64_t full_bar[kDStages], empty_bar[kDStages], tfull_bar, xch_bar;
  __shared__ unsigned tmem_base;
  __shared__ int abort_flag;
  __shared__ double red[16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = a.n, ne = (n + 1) >> 1, kbh = (ne + kDK - 1) / kDK, nts = (ne + kDN - 1) / kDN * (kDN / DN);
  const unsigned polls = a.polls ? a.polls : kDPolls;
  // rank 0 of the pair computes P, rank 1 Q
  const int rank = blockIdx.x & 1, nt = (blockIdx.x >> 1) % nts, mt = (blockIdx.x >> 1) / nts, m = blockIdx.y;
  if (!rhs_selected(a.st, a.mask, m)) return;  // uniform over the pair, before any set-up
  if (threadIdx.x == 0) {
    for (int s = 0; s < kDStages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(&tfull_bar, 1);
    mbar_init(&xch_bar, kDEpiWarps);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"((unsigned)(kSlices * DN))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  pair_arrive();  // the peer's barriers exist before the first arrival there (waited for below)
  const unsigned tmem = tmem_base;
  double acc[DN / 32] = {};  // (dot, out) over 8 columns each
  if (warp == 0) {
    // ---- MMA issuer ----
    if (lane == 0) {
      bool ok = true;
      for (int kb = 0; kb < kbh; ++kb) {
        const int s = kb % kDStages;
        if (!mbar_wait(&full_bar[s], (unsigned)(kb / kDStages) & 1u, polls)) {
          ok = false;
          break;
        }
        fence_after();
        unsigned char *st = dsm + s * T::stage;
#pragma unroll
        for (int j = 0; j < kDK / 16; ++j) {
          const uint64_t da = digit_desc(st + j * 256), db = digit_desc(st + kSlices * kDATile + j * 256);
          // an input slice against all its matrix slices: it stays in the tensor
          // core's collector buffer, and consecutive MMAs add to different sums
#pragma unroll
          for (int i = 0; i < kSlices; ++i) {
            const uint64_t ai = da + (uint64_t)(i * (kDATile >> 4));
            const unsigned add = (kb == 0 && j == 0 && i == 0) ? 0u : 1u;
#pragma unroll
            for (int t = 0; t < kSlices - i; ++t) {
              const uint64_t bt = db + (uint64_t)(t * (T::btile >> 4));
              const unsigned acc_t = tmem + (i + t) * DN;
              if (t == 0 && i < kSlices - 1) digit_mma<DN, 0>(acc_t, ai, bt, add);
              else if (t < kSlices - i - 1) digit_mma<DN, 1>(acc_t, ai, bt, add);
              else digit_mma<DN, 2>(acc_t, ai, bt, add);
            }
          }
        }
        digit_commit(&empty_bar[s]);
        if (kb == kbh - 1) digit_commit(&tfull_bar);
      }
      if (!ok) {
        atomicExch(&abort_flag, 1);
        if (a.err) atomicExch(a.err, 1);
      }
    }
    __syncwarp();
    pair_wait();
  } else if (warp == 1) {
    // ---- bulk copies ----
    if (lane == 0) {
      bool ok = true;
      int kb = 0;
      const unsigned char *ga = a.digits + (((size_t)m * a.mtiles + mt) * 2 + rank) * kbh * (size_t)(kSlices * kDATile);
      const unsigned char *gb = a.table + ((size_t)(nt * DN / kDN) * 2 + rank) * kbh * (size_t)(kSlices * kDBTile) +
                                nt * DN % kDN * (kDK * 2);
      for (; kb < kbh; ++kb) {
        const int s = kb % kDStages;
        if (kb >= kDStages && !mbar_wait(&empty_bar[s], (unsigned)(kb / kDStages - 1) & 1u, polls)) {
          ok = false;
          break;
        }
        if (abort_flag || kb == a.stall_at) {  // stall_at: test of the expiry path
          ok = false;
          break;
        }
        unsigned char *st = dsm + s * T::stage;
        mbar_arrive_tx(&full_bar[s], (unsigned)T::stage);
        bulk_g2s(st, ga + (size_t)kb * (kSlices * kDATile), kSlices * kDATile, &full_bar[s]);
        if constexpr (DN == kDN) {
          bulk_g2s(st + kSlices * kDATile, gb + (size_t)kb * (kSlices * kDBTile), kSlices * kDBTile, &full_bar[s]);
        } else {
          for (int t = 0; t < kSlices; ++t)
            bulk_g2s(st + kSlices * kDATile + t * T::btile, gb + ((size_t)kb * kSlices + t) * kDBTile, T::btile, &full_bar[s]);
        }
      }
      if (!ok) {
        atomicExch(&abort_flag, 1);
        if (a.err) atomicExch(a.err, 1);
        for (int j = kb > kDStages ? kb - kDStages : 0; j < kb; ++j)  // copies in flight (bounded)
          mbar_wait(&full_bar[j % kDStages], (unsigned)(j / kDStages) & 1u, polls);
      }
    }
    __syncwarp();
    pair_wait();
  } else if (warp < 4) {
    pair_wait();
  } else {
    // ---- epilogue: lane = row; warp w drains TMEM lane quarter w % 4.  The rank
    // finishes columns DN/2 rank .. + DN/2 - 1 of the tile, DN/4 per warp; first it
    // sends the peer what that needs for its columns ----
    pair_wait();
    constexpr int kOwn = DN / 4;
    const int q = warp & 3, half = (warp - 4) >> 2;
    const int trow = q * 32 + lane, row = mt * kDM + trow, l0 = nt * DN + rank * (DN / 2) + half * kOwn;
    const unsigned tw = tmem + ((unsigned)(q * 32) << 16) + half * kOwn;
    const bool row_ok = row < a.rows;
    bool good = true;
    // one lane polls: the tensor core reads its operands through the same port
    if (lane == 0) good = !abort_flag && mbar_wait(&tfull_bar, 0u, polls);
    good = __all_sync(0xffffffffu, good);
    double own[kOwn];
    if (good) {
      fence_after();
#pragma unroll
      for (int side = 0; side < 2; ++side) {  // the peer's columns, then this CTA's
        const unsigned tc = tw + (side == 0 ? 1 - rank : rank) * (DN / 2);
#pragma unroll
        for (int c8 = 0; c8 < kOwn / 8; ++c8) {
          unsigned D[kSlices][8];
#pragma unroll
          for (int d = 0; d < kSlices; ++d) tmem_ld8(tc + d * DN + c8 * 8, D[d]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            // V = sum_d D_d 128^(7-d)
            long long hi = __float2int_rn(__uint_as_float(D[0][i])), lo = __float2int_rn(__uint_as_float(D[4][i]));
#pragma unroll
            for (int d = 1; d < 4; ++d) {
              hi = hi * 128 + __float2int_rn(__uint_as_float(D[d][i]));
              lo = lo * 128 + __float2int_rn(__uint_as_float(D[4 + d][i]));
            }
            const double v = join(hi, lo);
            if (side == 0) peer_store(xch + (half * kOwn + c8 * 8 + i) * kDM + trow, v, rank ^ 1);
            else own[c8 * 8 + i] = v;
          }
        }
        if (side == 0) {
          asm volatile("fence.acq_rel.cluster;" ::: "memory");
          __syncwarp();
          if (lane == 0) peer_arrive(&xch_bar, rank ^ 1);
        }
      }
      if (lane == 0) good = peer_wait(&xch_bar, polls);
      good = __all_sync(0xffffffffu, good);
      asm volatile("fence.acq_rel.cluster;" ::: "memory");
    }
    if (!good) {  // the failure shows in the result too
      atomicExch(&abort_flag, 1);
      if (a.err) atomicExch(a.err, 1);
      if (row_ok)
        for (int j = 0; j < kOwn; ++j) {
          const int l = l0 + j, c0 = a.cosfwd ? 2 * l : l, c1 = a.cosfwd ? 2 * l + 1 : n - 1 - l;
          double *o = a.out + (size_t)m * (size_t)a.field + (size_t)row * a.pitch;
          if (l < ne) o[c0] = __longlong_as_double(0x7FF8000000000000ll);
          if (l < ne && c1 < n) o[c1] = __longlong_as_double(0x7FF8000000000000ll);
        }
    } else if (row_ok) {
      // out = V 2^sh: 2^(e - 55) 2^(eS - 54) 2^49 (the 8 highest of 15 digit
      // weights, 128^14 .. 128^7); a row that is not finite: NaN
      const double e = a.scale[(size_t)m * a.mtiles * kDM + row];
      const int sh = e == e ? (int)e + a.table_exp - 60 : 1 << 20;
      const size_t rb = (size_t)m * (size_t)a.field + (size_t)row * a.pitch;
      // 16-byte stores
      const bool even = ((a.pitch | (int)a.field) & 1) == 0 &&
                        ((reinterpret_cast<uintptr_t>(a.out) | reinterpret_cast<uintptr_t>(a.dot)) & 15) == 0;
      auto put = [&](int col, double v, double &acc) {
        if (a.dot != nullptr) acc = fma(a.dot[rb + col], v, acc);
        a.out[rb + col] = v;
      };
      auto put2 = [&](int col, double u, double v, double &acc) {
        if (!even) {
          put(col, u, acc);
          put(col + 1, v, acc);
          return;
        }
        if (a.dot != nullptr) {
          const double2 rv = *reinterpret_cast<const double2 *>(a.dot + rb + col);
          acc = fma(rv.x, u, acc);
          acc = fma(rv.y, v, acc);
        }
        *reinterpret_cast<double2 *>(a.out + rb + col) = make_double2(u, v);
      };
#pragma unroll
      for (int i = 0; i < kOwn; i += 2) {
        const int l = l0 + i;
        double &sum = acc[i / 8];
        double o[2][2];  // [column l, l + 1][run]
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const double other = xch[(half * kOwn + i + j) * kDM + trow];
          const double p = rank == 0 ? own[i + j] : other, v = rank == 0 ? other : own[i + j];
          o[j][0] = scaled(a.cosfwd ? p : p + v, sh);
          o[j][1] = scaled(a.cosfwd ? v : p - v, sh);
        }
        if (a.cosfwd) {  // columns 2 l .. 2 l + 3
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int c = 2 * (l + j);
            if (l + j >= ne) continue;
            if (c + 1 < n) put2(c, o[j][0], o[j][1], sum);
            else put(c, o[j][0], sum);
          }
        } else if (l + 1 < ne && (n & 1) == 0) {
          put2(l, o[0][0], o[1][0], sum);
          put2(n - 2 - l, o[1][1], o[0][1], sum);
        } else {
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (l + j >= ne) continue;
            put(l + j, o[j][0], sum);
            if (n - 1 - l - j != l + j) put(n - 1 - l - j, o[j][1], sum);  // the middle column of odd n once
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  pair_arrive();  // the peer writes into this CTA's shared memory until here
  pair_wait();
  if (warp == 0) {
    if (abort_flag) mbar_wait(&tfull_bar, 0u, polls);  // a bounded moment for MMAs in flight
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((unsigned)(kSlices * DN))
                 : "memory");
  }
  if (a.dot != nullptr) {
    // a partial per 128 rows x 16 columns, from 8 warp sums in a fixed order
    constexpr int parts = DN / 32;
    if (warp >= 4) {
#pragma unroll
      for (int g = 0; g < parts; ++g) {
        const double w = warp_sum(acc[g]);
        if (lane == 0) red[((warp - 4) >> 2) * parts * 4 + g * 4 + (warp & 3)] = w;
      }
    }
    __syncthreads();
    double *part = a.partial + (size_t)m * kPartialStride;
    if (threadIdx.x < parts) {
      double sum = 0.0;
      for (int i = 0; i < 8; ++i) sum += red[threadIdx.x * 8 + i];
      part[blockIdx.x * parts + threadIdx.x] = sum;
    }
    __syncthreads();
    finish_rhs(a.fin, m, gridDim.x, part, (int)gridDim.x * parts, red);
  }
}

// Numbers as pairs of FP64 numbers, v = h + l, for the matrix entries (two-sum and
// two-product; some 100 bits).
struct Pair {
  double h, l;
};
__device__ __forceinline__ Pair pair_sum(double a, double b) {
  const double s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
  const Pair s = pair_sum(a.h, b.h);
  return pair_sum(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  const double p = a.h * b.h;
  return pair_sum(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
__device__ __forceinline__ Pair pair_div(Pair a, double d) {
  const double q = a.h / d;
  return pair_sum(q, (fma(-q, d, a.h) + a.l) / d);
}

// t[j] = sin(pi j / den), j <= den / 2, by the Taylor series of the sine or cosine of at
// most pi / 4.  FP64 functions would leave an error of about 2^-53 in every entry of the
// matrix, and the argument's rounding one that neighbouring entries share: it showed in
// constant rows (511 columns: 4.3 2^-53 of the row's norm; now 0.8).
__global__ void __launch_bounds__(128) sine_list_kernel(Pair *t, int den) {
  const int j = blockIdx.x * 128 + threadIdx.x;
  if (j > den / 2) return;
  const bool co = 4 * j > den;  // cos(pi (den - 2 j) / (2 den))
  const Pair x = pair_mul(pair_div(Pair{co ? (double)(den - 2 * j) : (double)j, 0.0}, co ? 2.0 * den : (double)den),
                          Pair{3.14159265358979312, 1.2246467991473532e-16});
  const Pair x2 = pair_mul(x, x);
  Pair term = co ? Pair{1.0, 0.0} : x, sum = term;
  for (int k = co ? 1 : 2; k < 24; k += 2) {  // -x^2 / (k (k + 1))
    term = pair_div(pair_mul(term, x2), -(double)(k * (k + 1)));
    sum = pair_add(sum, term);
  }
  t[j] = sum;
}

// Matrix digits: tiles (N tile, K block, slice) as the stages copy them; row l of a
// tile the output column, k the position of the half.  sine: sine_list_kernel's, of
// den = n + 1 for the sine, 2 n for the cosines.
__global__ void __launch_bounds__(256) digit_table_kernel(unsigned char *__restrict__ t, const Pair *__restrict__ sine,
                                                          int n, int kind, int e) {
  const int ne = (n + 1) >> 1, kbh = (ne + kDK - 1) / kDK, nts = (ne + kDN - 1) / kDN, L = n + 1;
  const size_t total = (size_t)nts * 2 * kbh * kDN * kDK;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int kl = (int)(i % kDK), nl = (int)(i / kDK % kDN), kb = (int)(i / (kDK * kDN) % (2 * kbh));
    const int nt = (int)(i / ((size_t)kDK * kDN * 2 * kbh));
    const bool second = kb >= kbh;
    const int l = nt * kDN + nl, kk = (second ? kb - kbh : kb) * kDK + kl;
    Pair v{0.0, 0.0};
    if (l < ne && kk < ne) {
      // sqrt(num / den) c, the angles of c reduced exactly
      auto entry = [&](int num, int den, Pair c) {
        const Pair q = pair_div(Pair{(double)num, 0.0}, (double)den);
        const double r = sqrt(q.h);
        v = pair_mul(c, Pair{r, (fma(-r, r, q.h) + q.l) / (2.0 * r)});
      };
      auto sign = [](Pair c, bool minus) { return minus ? Pair{-c.h, -c.l} : c; };
      // orthonormal cosine entry of mode f at node k, cos(pi m / (2 n)) = sin(pi (n - m) / (2 n))
      auto cosm = [&](int f, int k) {
        int m = (int)((long long)(2 * k + 1) * f % (4LL * n));
        if (m > 2 * n) m = 4 * n - m;
        const bool minus = m > n;
        if (minus) m = 2 * n - m;
        entry(f == 0 ? 1 : 2, n, sign(sine[n - m], minus));
      };
      if (kind == kTableCosForward) {
        const int f = second ? 2 * l + 1 : 2 * l;
        if (f < n) cosm(f, kk);
      } else {
        const int k = second ? 2 * kk + 1 : 2 * kk;
        if (k < n) {
          if (kind == kTableCosInverse) {
            cosm(k, l);
          } else {
            int m = (int)((long long)(k + 1) * (l + 1) % (2LL * L));
            const bool minus = m > L;
            if (minus) m -= L;
            entry(2, L, sign(sine[m > L - m ? L - m : m], minus));
          }
        }
      }
    }
    // v 2^(54 - e) rounded to an integer
    const double w = ldexp(v.h, 54 - e);
    const long long X = llrint(w);
    float d[kSlices];
    digits_of(X + llrint((w - (double)X) + ldexp(v.l, 54 - e)), d);
    unsigned char *p = t + ((size_t)nt * 2 * kbh + kb) * (size_t)(kSlices * kDBTile) + digit_byte(nl, kl);
#pragma unroll
    for (int s = 0; s < kSlices; ++s)
      *reinterpret_cast<__nv_bfloat16 *>(p + s * kDBTile) = __float2bfloat16(d[s]);
  }
}

}  // namespace

bool digits_apply(int rows, int n) {
  return n >= kDigitMinN && n <= kDigitMaxN && rows >= (n <= 512 ? kDigitMinRows : kDigitMinRowsLong) &&
         rows <= kDigitMaxRows;
}
int digit_mtiles(int rows) { return (rows + kDM - 1) / kDM; }
size_t digit_bytes(int rows, int n) {
  const int ne = (n + 1) >> 1, kbh = (ne + kDK - 1) / kDK;
  return (size_t)digit_mtiles(rows) * 2 * kbh * kSlices * kDATile;
}
int digit_table_exp(int n, int kind) {
  // largest entry at most sqrt(2 / (n + 1)) or sqrt(2 / n)
  return (int)std::floor(std::log2(std::sqrt(2.0 / (kind == kTableSine ? n + 1 : n))));
}
int digit_split_blocks(int rows) { return (rows + 7) / 8; }
// Partials of (dot, out) per right-hand side: by its sizes alone, whatever the
// tiles, so that results do not depend on how many share a launch.
int digit_gemm_partials(int rows, int n) { return 4 * digit_mtiles(rows) * (((n + 1) / 2 + kDN - 1) / kDN); }

// Digits of the transform matrix per (device, n, kind), kept for the life of the
// process like the BF16 tables.
const unsigned char *digit_table(int device, int n, int kind, cudaStream_t s, bool make) {
  static std::mutex mu;
  static std::vector<std::pair<long long, unsigned char *>> tables;
  std::lock_guard<std::mutex> lock(mu);
  const long long key = (long long)device << 32 | (unsigned)n | (long long)kind << 24;
  for (auto &e : tables)
    if (e.first == key) return e.second;
  if (!make) return nullptr;
  const int ne = (n + 1) >> 1, kbh = (ne + kDK - 1) / kDK, nts = (ne + kDN - 1) / kDN;
  const size_t bytes = (size_t)nts * 2 * kbh * kSlices * kDBTile;
  // the matrix and, behind it, the list of sines it is made from
  const int den = kind == kTableSine ? n + 1 : 2 * n;
  unsigned char *d = nullptr;
  if (cudaMalloc((void **)&d, bytes + (den / 2 + 1) * sizeof(Pair)) != cudaSuccess) return nullptr;
  Pair *sine = reinterpret_cast<Pair *>(d + bytes);
  note_launch();
  sine_list_kernel<<<den / 256 + 1, 128, 0, s>>>(sine, den);
  note_launch();
  digit_table_kernel<<<608, 256, 0, s>>>(d, sine, n, kind, digit_table_exp(n, kind));
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
    cudaFree(d);
    return nullptr;
  }
  tables.push_back({key, d});
  return d;
}

void launch_digit_split(const DigitArgs &a, cudaStream_t s) {
  note_launch();
  digit_split_kernel<<<dim3(digit_split_blocks(a.rows), a.m), 256, 0, s>>>(a);
}

template <int DN>
static void digit_gemm_launch(const DigitArgs &a, cudaStream_t s) {
  ensure_smem_attr((const void *)digit_gemm_kernel<DN>, DigitTile<DN>::smem);
  digit_gemm_kernel<DN><<<dim3(digit_gemm_partials(a.rows, a.n) * 32 / DN, a.m), kDThreads, DigitTile<DN>::smem, s>>>(a);
}

// Output columns per CTA (the results are the same): 64, or 32 where 64 would leave
// more than half of the SMs without a CTA.  An MMA of 32 columns takes 45 cycles, one
// of 64 takes 50, and the input digits are copied for each: 500 rows of 511 take
// 6 us less, 4000 rows 20 us more.
void launch_digit_gemm(const DigitArgs &a, cudaStream_t s) {
  note_launch();
  if (a.m * digit_gemm_partials(a.rows, a.n) / 2 > 76) digit_gemm_launch<64>(a, s);
  else digit_gemm_launch<32>(a, s);
}

}  // namespace ax
