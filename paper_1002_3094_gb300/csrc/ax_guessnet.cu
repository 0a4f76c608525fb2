// Initial-guess network: a small convolutional encoder-decoder that maps
// (log kappa, q, f / s) on an H x W lattice to u0 / s, trained on solutions
// that the solver itself produced.  The paper has no such component; it is
// the learned warm start of the production form: the CG solve always starts
// from it only if it lowers the initial residual, and always iterates to the
// same tolerance.
//
// Inputs [B][3][H][W] (NCHW, FP32) and outputs [B][H][W]; activations between
// layers in BF16, gradients in FP32 (see Layouts below).  Conv weights
// [3][3][Cin][Cout] ([dy+1][dx+1][ci][co], "same" cross-correlation with zero
// padding), FP32 master copy + packed BF16 compute copies; FP32 accumulation
// everywhere.
//
// Architecture (levels H, H/2, H/4, H/8; channels c1..c4):
//   e1a e1b | pool | e2a e2b | pool | e3a e3b | pool | b1 b2 | up |
//   d3a(+skip e3b) d3b | up | d2a(+skip e2b) d2b | up | d1a(+skip e1b) d1b | head(1x1)
// Every 3x3 conv is followed by ReLU; the "+skip" layers add the encoder
// activation of the same level after their ReLU.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "ax_common.cuh"

namespace ax {
namespace {

using bf16 = __nv_bfloat16;

// ---------------------------------------------------------------------------
// Layouts.  Activations are NHWC BF16, channels padded to a multiple of 8 (16
// bytes; the padding holds zeros); gradients are NHWC FP32 with the same padding
// (written as zeros).  Convolutions are implicit GEMMs on the tensor cores,
// mma.sync m16n8k16 (BF16 x BF16 -> FP32): the 3 x 3 taps and chunks of 16 input
// channels form K.  Weights are kept packed per layer as [chunk of 16 k][tap]
// [n][16 k] BF16, once for the forward pass (n = output, k = input channel) and
// once, taps flipped, for the backward-data pass (n = input, k = output).
// FP32 gradients enter the tensor cores as three BF16 numbers, g = h + m + l
// (24 bits: all of an FP32 significand), so that products and sums keep FP32
// accuracy.
// ---------------------------------------------------------------------------
__host__ __device__ inline int pad8(int c) { return (c + 7) & ~7; }
__host__ __device__ inline int chunks16(int c) { return (c + 15) >> 4; }

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(unsigned addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(unsigned addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm2(unsigned addr, unsigned &r0, unsigned &r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void ldsm2t(unsigned addr, unsigned &r0, unsigned &r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Byte offset of the 16-byte half `half` of 32-byte row `row` in a shared array
// of such rows: the halves are swapped in every other group of 4 rows, so that
// the 8 rows an ldmatrix phase reads fall in distinct banks.
__device__ __forceinline__ unsigned row32(int row, int half) {
  return (unsigned)(row * 32 + ((half ^ ((row >> 2) & 1)) << 4));
}

// a + b as three BF16 pairs: the high, middle and low parts (each the rounding
// of what the ones before left).
__device__ __forceinline__ void split3(float a, float b, unsigned &h, unsigned &m, unsigned &l) {
  h = bf16_pack2(a, b);
  const float ra = a - bf16_lo(h), rb = b - bf16_hi(h);
  m = bf16_pack2(ra, rb);
  l = bf16_pack2(ra - bf16_lo(m), rb - bf16_hi(m));
}

// ---------------------------------------------------------------------------
// 3 x 3 convolution.  A CTA computes a patch of 8 MW rows x 16 pixels (warp w: MW
// rows of 16 pixels) for 8 NT output channels; K runs over chunks of 16 channels
// and, inside, the 9 taps.  Shared memory holds the haloed patch as [pixel][16
// channels] and the chunk's weights as [tap][n][16], rows of 32 bytes read with
// ldmatrix.  What bounds it is the tensor pipe once each fragment feeds several
// MMAs: per tap MW + NT / 2 ldmatrix for MW NT MMAs (the kernel before read 12
// words per lane for 4 MMAs of a 16 x 32 warp tile and converted its input
// element by element: 45 TFLOP/s at 256 x 256, batch 16).
//   PLANES = 1: BF16 input, forward: out = relu(conv + bias), out2 = out + skip.
//     The order of accumulation (chunk, then tap) is that of the plain sum over K.
//   PLANES = 3: FP32 input split in three, backward data: out = conv (* the
//     ReLU mask of act), out2 = conv unmasked.  The tensor core's accumulation
//     truncates (emptied once per chunk of 27 products, the gradients of all
//     layers were 7e-7 off 64 bits against 3e-7 for FP32 FMAs), so every tap's
//     products, the small parts first, go to a fresh accumulator that is added to
//     the sum in FP32.
// ---------------------------------------------------------------------------
struct ConvArgs {
  const void *in;       // [B][H >> up][W >> up][pad8(Cin)]
  const bf16 *w;        // packed [chunk][9][n8][16]
  const float *bias;    // forward
  void *out;            // BF16 (forward) or FP32 [B][H][W][pad8(Cout)]
  void *out2;           // second output or null
  const bf16 *skip;     // forward with out2: added after the ReLU
  const bf16 *mask;     // backward: activation whose sign masks out (null: none)
  int cin, cout, H, W, up;
};
template <int NT, int MW, int PLANES>
struct ConvShape {
  static constexpr int rows = 8 * MW + 2, pix = rows * 18;
  static constexpr int in_bytes = pix * 32 * PLANES;
  static constexpr int w_bytes = 9 * 8 * NT * 32;
  static constexpr int stages = PLANES == 1 ? 2 : 1;
  static constexpr int smem = stages * (in_bytes + w_bytes);
};

template <int NT, int MW, int PLANES>
__global__ void __launch_bounds__(256, 2) conv3x3_kernel(const ConvArgs a) {
  using S = ConvShape<NT, MW, PLANES>;
  extern __shared__ __align__(128) unsigned char csm[];
  const int H = a.H, W = a.W, up = a.up;
  const int tiles_x = (W + 15) >> 4;
  const int x0 = (blockIdx.x % tiles_x) * 16, y0 = (blockIdx.x / tiles_x) * 8 * MW;
  const int n0 = blockIdx.y * 8 * NT;
  const int b = blockIdx.z;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int cpin = pad8(a.cin), n8 = pad8(a.cout);
  const int Hs = H >> up, Ws = W >> up;
  const int nchunk = chunks16(a.cin);
  auto in_at = [&](int s) { return smem_u32(csm) + s * (S::in_bytes + S::w_bytes); };
  auto w_at = [&](int s) { return in_at(s) + S::in_bytes; };
  auto load_w = [&](int s, int k) {
    for (int e = t; e < 9 * 8 * NT * 2; e += 256) {
      const int half = e & 1, r = e >> 1, tap = r / (8 * NT), n = r - tap * 8 * NT;
      const bool ok = n0 + n < n8;
      cp_async16(w_at(s) + row32(r, half),
                 a.w + (ok ? ((((size_t)k * 9 + tap) * n8 + n0 + n) * 16 + half * 8) : 0), ok);
    }
  };
  auto load_in = [&](int s, int k) {  // PLANES == 1
    const bf16 *in = static_cast<const bf16 *>(a.in) + (size_t)b * Hs * Ws * cpin;
    for (int e = t; e < S::pix * 2; e += 256) {
      const int half = e & 1, p = e >> 1, yy = p / 18, xx = p - yy * 18;
      const int gy = y0 + yy - 1, gx = x0 + xx - 1, c = k * 16 + half * 8;
      const bool ok = gy >= 0 && gy < H && gx >= 0 && gx < W && c < cpin;
      cp_async16(in_at(s) + row32(p, half), in + (ok ? ((size_t)(gy >> up) * Ws + (gx >> up)) * cpin + c : 0), ok);
    }
  };
  auto load_split = [&](int k) {  // PLANES == 3
    const float *in = static_cast<const float *>(a.in) + (size_t)b * H * W * cpin;
    for (int e = t; e < S::pix * 2; e += 256) {
      const int half = e & 1, p = e >> 1, yy = p / 18, xx = p - yy * 18;
      const int gy = y0 + yy - 1, gx = x0 + xx - 1, c = k * 16 + half * 8;
      float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
      if (gy >= 0 && gy < H && gx >= 0 && gx < W && c < cpin) {
        const float4 *src = reinterpret_cast<const float4 *>(in + ((size_t)gy * W + gx) * cpin + c);
        u = src[0];
        v = src[1];
      }
      uint4 h, m, l;
      split3(u.x, u.y, h.x, m.x, l.x);
      split3(u.z, u.w, h.y, m.y, l.y);
      split3(v.x, v.y, h.z, m.z, l.z);
      split3(v.z, v.w, h.w, m.w, l.w);
      unsigned char *dst = csm + row32(p, half);
      *reinterpret_cast<uint4 *>(dst) = h;
      *reinterpret_cast<uint4 *>(dst + S::pix * 32) = m;
      *reinterpret_cast<uint4 *>(dst + 2 * S::pix * 32) = l;
    }
  };
  float sum[MW][NT][4];
#pragma unroll
  for (int i = 0; i < MW; ++i)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int c = 0; c < 4; ++c) sum[i][n][c] = 0.f;
  // one chunk's products into the sums
  auto products = [&](int s) {
    const unsigned ib = in_at(s), wb = w_at(s);
    // ldmatrix row of this lane: A rows (pixels) lane & 15, half lane >> 4; B rows
    // (channels) (lane & 7) + 8 (lane >> 4), half (lane >> 3) & 1
    const int ap = lane & 15, ah = lane >> 4, bn = (lane & 7) + ((lane >> 4) << 3), bh = (lane >> 3) & 1;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int dy = tap / 3, dx = tap % 3;
      unsigned bf[NT][2];
#pragma unroll
      for (int n = 0; n + 1 < NT; n += 2) {
        unsigned r[4];
        ldsm4(wb + row32(tap * 8 * NT + n * 8 + bn, bh), r);
        bf[n][0] = r[0]; bf[n][1] = r[1]; bf[n + 1][0] = r[2]; bf[n + 1][1] = r[3];
      }
      if (NT & 1) ldsm2(wb + row32(tap * 8 * NT + (NT - 1) * 8 + (lane & 7), (lane >> 3) & 1), bf[NT - 1][0], bf[NT - 1][1]);
#pragma unroll
      for (int i = 0; i < MW; ++i) {
        const int p = (warp * MW + i + dy) * 18 + dx + ap;
        if constexpr (PLANES == 1) {
          unsigned af[4];
          ldsm4(ib + row32(p, ah), af);
#pragma unroll
          for (int n = 0; n < NT; ++n) mma_bf16_16816(sum[i][n], af, bf[n][0], bf[n][1]);
        } else {
          unsigned af[PLANES][4];
#pragma unroll
          for (int q = 0; q < PLANES; ++q) ldsm4(ib + q * S::pix * 32 + row32(p, ah), af[q]);
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int q = PLANES - 1; q >= 0; --q) mma_bf16_16816(acc, af[q], bf[n][0], bf[n][1]);
#pragma unroll
            for (int c = 0; c < 4; ++c) sum[i][n][c] += acc[c];
          }
        }
      }
    }
  };
  if constexpr (PLANES == 1) {
    load_in(0, 0);
    load_w(0, 0);
    cp_async_commit();
    for (int k = 0; k < nchunk; ++k) {
      if (k + 1 < nchunk) {
        load_in((k + 1) & 1, k + 1);
        load_w((k + 1) & 1, k + 1);
        cp_async_commit();
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
      products(k & 1);
      __syncthreads();
    }
  } else {
    for (int k = 0; k < nchunk; ++k) {
      load_w(0, k);
      cp_async_commit();
      load_split(k);
      cp_async_wait<0>();
      __syncthreads();
      products(0);
      __syncthreads();
    }
  }
  // epilogue: sum[i][n][0..1] pixel g, channels n*8 + 2 tq + {0, 1}; [2..3] pixel g + 8
  const int g = lane >> 2, tq = lane & 3;
#pragma unroll
  for (int i = 0; i < MW; ++i) {
    const int y = y0 + warp * MW + i;
    if (y >= H) continue;
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int x = x0 + g + 8 * hf;
      if (x >= W) continue;
      const size_t pix = ((size_t)b * H + y) * W + x;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const int co = n0 + n * 8 + 2 * tq;
        if (co >= n8) continue;
        const size_t o = pix * n8 + co;
        float v0 = sum[i][n][2 * hf], v1 = sum[i][n][2 * hf + 1];
        if constexpr (PLANES == 1) {
          // padding channels (their weights are zero) stay zero
          v0 = co < a.cout ? fmaxf(v0 + a.bias[co], 0.f) : 0.f;
          v1 = co + 1 < a.cout ? fmaxf(v1 + a.bias[co + 1], 0.f) : 0.f;
          *reinterpret_cast<unsigned *>(static_cast<bf16 *>(a.out) + o) = bf16_pack2(v0, v1);
          if (a.out2 != nullptr) {
            const unsigned s = *reinterpret_cast<const unsigned *>(a.skip + o);
            *reinterpret_cast<unsigned *>(static_cast<bf16 *>(a.out2) + o) =
                bf16_pack2(v0 + bf16_lo(s), v1 + bf16_hi(s));
          }
        } else {
          if (a.out2 != nullptr) *reinterpret_cast<float2 *>(static_cast<float *>(a.out2) + o) = make_float2(v0, v1);
          if (a.mask != nullptr) {
            const unsigned s = *reinterpret_cast<const unsigned *>(a.mask + o);
            v0 = bf16_lo(s) > 0.f ? v0 : 0.f;
            v1 = bf16_hi(s) > 0.f ? v1 : 0.f;
          }
          *reinterpret_cast<float2 *>(static_cast<float *>(a.out) + o) = make_float2(v0, v1);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Weight gradient of a 3 x 3 convolution,
//   dW[tap][ci][co] = sum over pixels of in[pixel + tap][ci] gz[pixel][co],
// as a GEMM on the tensor cores with M = 16 input channels, N = 24 output
// channels and K = pixels; both operands are read transposed (ldmatrix.trans)
// from their NHWC tiles.  A warp keeps all 9 taps' accumulators (108 registers):
// each k block of 16 pixels takes 9 ldmatrix of the input (the taps' shifts) and
// feeds 81 MMAs (9 taps x 3 n-tiles x the 3 BF16 parts of gz).  A CTA owns one
// (ci, co) block and every gridDim.z-th 16 x 16 pixel tile, warp w the rows 2 w,
// 2 w + 1; the next tile is loaded while one is multiplied.  The truncating
// accumulators are emptied into FP32 sums after every tile (18 products per
// element).  The warps' sums are added in order and written as one partial per
// CTA: deterministic.  (Before: FP32 FMAs on CUDA cores, one partial per 32 x 32
// tile, 18 ms of a 256 x 256 batch-16 step.)
// ---------------------------------------------------------------------------
constexpr int kWgN = 24;                       // output channels per CTA
constexpr int kWgIn = 18 * 18 * 32;            // input tile bytes (16 channels)
constexpr int kWgG = 256 * kWgN * 2;           // bytes of one part of the gz tile
constexpr int kWgSmem = 2 * kWgIn + 3 * kWgG;

struct WgradArgs {
  const bf16 *in;      // [B][H >> up][W >> up][cpin]
  const float *gz;     // [B][H][W][pad8(cout)]
  float *partial;      // [gridDim.z][9][cin][cout]
  int cin, cpin, cout, B, H, W, up;
};
__global__ void __launch_bounds__(256, 1) conv3x3_wgrad_kernel(const WgradArgs a) {
  extern __shared__ __align__(128) unsigned char wsm[];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int ci0 = blockIdx.x * 16, co0 = blockIdx.y * kWgN;
  const int H = a.H, W = a.W, up = a.up, Hs = H >> up, Ws = W >> up, cpo = pad8(a.cout);
  const int tx = (W + 15) >> 4, ty = (H + 15) >> 4, ntile = a.B * tx * ty;
  const unsigned sin0 = smem_u32(wsm), sg = sin0 + 2 * kWgIn;
  auto load_in = [&](int s, int tile) {
    const int b = tile / (tx * ty), r = tile - b * tx * ty;
    const int y0 = (r / tx) * 16, x0 = (r % tx) * 16;
    const bf16 *in = a.in + (size_t)b * Hs * Ws * a.cpin;
    for (int e = t; e < 18 * 18 * 2; e += 256) {
      const int half = e & 1, p = e >> 1, yy = p / 18, xx = p - yy * 18;
      const int gy = y0 + yy - 1, gx = x0 + xx - 1, c = ci0 + half * 8;
      const bool ok = gy >= 0 && gy < H && gx >= 0 && gx < W && c < a.cpin;
      cp_async16(sin0 + s * kWgIn + row32(p, half),
                 in + (ok ? ((size_t)(gy >> up) * Ws + (gx >> up)) * a.cpin + c : 0), ok);
    }
    cp_async_commit();
  };
  float4 gv[6];  // the tile's gz: 256 pixels x 6 groups of 4 channels over 256 threads
  auto load_g = [&](int tile) {
    const int b = tile / (tx * ty), r = tile - b * tx * ty;
    const int y0 = (r / tx) * 16, x0 = (r % tx) * 16;
    const float *g = a.gz + (size_t)b * H * W * cpo;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const int e = t + j * 256, p = e / 6, c = co0 + (e - p * 6) * 4;
      const int gy = y0 + (p >> 4), gx = x0 + (p & 15);
      gv[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (gy < H && gx < W && c < cpo) gv[j] = *reinterpret_cast<const float4 *>(g + ((size_t)gy * W + gx) * cpo + c);
    }
  };
  auto store_g = [&]() {
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const int e = t + j * 256, p = e / 6, q = e - p * 6;
      uint2 h, m, l;
      split3(gv[j].x, gv[j].y, h.x, m.x, l.x);
      split3(gv[j].z, gv[j].w, h.y, m.y, l.y);
      unsigned char *dst = wsm + 2 * kWgIn + p * (kWgN * 2) + q * 8;
      *reinterpret_cast<uint2 *>(dst) = h;
      *reinterpret_cast<uint2 *>(dst + kWgG) = m;
      *reinterpret_cast<uint2 *>(dst + 2 * kWgG) = l;
    }
  };
  float sum[9][3][4];
#pragma unroll
  for (int i = 0; i < 9; ++i)
#pragma unroll
    for (int n = 0; n < 3; ++n)
#pragma unroll
      for (int c = 0; c < 4; ++c) sum[i][n][c] = 0.f;
  int tile = blockIdx.z, s = 0;
  if (tile < ntile) {
    load_in(0, tile);
    load_g(tile);
  }
  for (; tile < ntile; tile += gridDim.z, s ^= 1) {
    store_g();
    const int next = tile + gridDim.z;
    if (next < ntile) {
      load_in(s ^ 1, next);
      load_g(next);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    // B parts of this warp's two k blocks; lanes 0-15 address the rows (pixels)
    unsigned bfr[2][3][3][2];
#pragma unroll
    for (int kb = 0; kb < 2; ++kb)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const unsigned base = sg + q * kWgG + ((warp * 2 + kb) * 16 + (lane & 15)) * (kWgN * 2);
        unsigned r[4];
        ldsm4t(base + (lane >> 4) * 16, r);  // n-tiles 0 and 1
        bfr[kb][q][0][0] = r[0]; bfr[kb][q][0][1] = r[1]; bfr[kb][q][1][0] = r[2]; bfr[kb][q][1][1] = r[3];
        ldsm2t(base + 32, bfr[kb][q][2][0], bfr[kb][q][2][1]);
      }
    const unsigned ib = sin0 + s * kWgIn;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int dy = tap / 3, dx = tap % 3;
      float acc[3][4];
#pragma unroll
      for (int n = 0; n < 3; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[n][c] = 0.f;
#pragma unroll
      for (int kb = 0; kb < 2; ++kb) {
        // A (16 ci x 16 pixels) from [pixel][ci]: matrices (k 0-7, m 0-7),
        // (k 0-7, m 8-15), (k 8-15, m 0-7), (k 8-15, m 8-15), transposed
        const int p = (warp * 2 + kb + dy) * 18 + dx + (lane & 7) + ((lane >> 4) << 3);
        unsigned af[4];
        ldsm4t(ib + row32(p, (lane >> 3) & 1), af);
#pragma unroll
        for (int q = 2; q >= 0; --q)
#pragma unroll
          for (int n = 0; n < 3; ++n) mma_bf16_16816(acc[n], af, bfr[kb][q][n][0], bfr[kb][q][n][1]);
      }
#pragma unroll
      for (int n = 0; n < 3; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) sum[tap][n][c] += acc[n][c];
    }
    __syncthreads();
  }
  // the 8 warps' sums in order (the tiles' shared memory is free now)
  float *red = reinterpret_cast<float *>(wsm);
  for (int w = 0; w < 8; ++w) {
    if (warp == w) {
#pragma unroll
      for (int i = 0; i < 9; ++i)
#pragma unroll
        for (int n = 0; n < 3; ++n)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float *r = red + ((i * 3 + n) * 4 + c) * 32 + lane;
            *r = (w == 0 ? 0.f : *r) + sum[i][n][c];
          }
    }
    __syncthreads();
  }
  float *pp = a.partial + (size_t)blockIdx.z * 9 * a.cin * a.cout;
  for (int e = t; e < 9 * 16 * kWgN; e += 256) {
    const int tap = e / (16 * kWgN), r = e - tap * 16 * kWgN, ci = r / kWgN, co = r - ci * kWgN;
    if (ci0 + ci >= a.cin || co0 + co >= a.cout) continue;
    // element (row ci, column co) of the accumulator tile: rows g and g + 8 in
    // registers {0, 1} and {2, 3}, columns 2 tq + {0, 1}
    const int n = co >> 3, cc = ((ci >> 3) << 1) | (co & 1), ln = ((ci & 7) << 2) | ((co & 7) >> 1);
    pp[((size_t)tap * a.cin + ci0 + ci) * a.cout + co0 + co] = red[((tap * 3 + n) * 4 + cc) * 32 + ln];
  }
}

// out[i] = sum over the slots of partial[slot][i] (a fixed order: 8 groups of
// slots in FP32, then the groups).  With planes = 3 (the network's FP32 input as
// three BF16 planes of 3 channels) the three planes' rows of a partial,
// [9][9][cout], add up to [9][3][cout].  256 threads: 32 elements x 8 groups (one
// thread per element left most of the chip idle over a chain of up to 304
// loads: 17 us on average, 30 launches per step).
__global__ void __launch_bounds__(256) sum_partials(const float *__restrict__ partial, int slots, size_t n,
                                                    float *__restrict__ out, int planes, int cout) {
  __shared__ float red[8][32];
  const size_t i = blockIdx.x * (size_t)32 + (threadIdx.x & 31);
  const int grp = threadIdx.x >> 5;
  float s = 0.f;
  if (i < n) {
    if (planes == 1) {
#pragma unroll 8
      for (int k = grp; k < slots; k += 8) s += partial[(size_t)k * n + i];
    } else {
      const size_t co = i % cout, r = i / cout, ci = r % 3, tap = r / 3;
#pragma unroll 4
      for (int k = grp; k < slots; k += 8) {
        const float *p = partial + (size_t)k * 3 * n + (tap * 9 + ci) * cout + co;
        s += (p[0] + p[3 * (size_t)cout]) + p[6 * (size_t)cout];
      }
    }
  }
  red[grp][threadIdx.x & 31] = s;
  __syncthreads();
  if (grp == 0 && i < n) {
    float tot = red[0][threadIdx.x];
#pragma unroll
    for (int g = 1; g < 8; ++g) tot += red[g][threadIdx.x];
    out[i] = tot;
  }
}

// s[t][.] += s[t + k q][.] over the `groups` groups of q threads, in a fixed order; the
// first group holds the result.  Every thread of the block calls it.
template <int N>
__device__ __forceinline__ void add_groups(Sum3 (*s)[N], int q, int groups) {
  const int grp = threadIdx.x / q;
  for (int left = groups; left > 1;) {
    const int half = (left + 1) >> 1;
    if (grp < left - half)
#pragma unroll
      for (int i = 0; i < N; ++i) s[threadIdx.x][i].add(s[threadIdx.x + half * q][i]);
    __syncthreads();
    left = half;
  }
}

// out[i] = sum over the slots of partial[slot][i], rounded to FP32 once.  (The sums of
// gradients cancel: rounded to FP32 per block, 912 of them, they were some 100 times as
// far off as the plane sums in FP64 before.)  256 threads: 8 elements x 32 groups of
// slots, added in a fixed order.
__global__ void __launch_bounds__(256) sum_sum3(const Sum3 *__restrict__ partial, int slots, int n,
                                                float *__restrict__ out) {
  __shared__ Sum3 red[256][1];
  const int i = blockIdx.x * 8 + (threadIdx.x & 7);
  Sum3 s;
  if (i < n) {
#pragma unroll 8
    for (int k = threadIdx.x >> 3; k < slots; k += 32) s.add(partial[(size_t)k * n + i]);
  }
  red[threadIdx.x][0] = s;
  __syncthreads();
  add_groups(red, 8, 32);
  if (threadIdx.x < 8 && i < n) out[i] = red[threadIdx.x][0].value();
}

// Per-block sums of gz over pixels, per channel: partial[block][c].  blockDim = 256:
// groups of cp / 4 threads walk the pixels, 4 channels each.
__global__ void __launch_bounds__(256) channel_sums(const float *__restrict__ g, int C, int cp, size_t pixels,
                                                    Sum3 *__restrict__ partial) {
  __shared__ Sum3 sd[256][4];
  const int q = cp / 4, groups = max(1, 256 / q);
  // channels beyond what one pass of the threads covers are taken in turn
  for (int c0 = 0; c0 < q; c0 += 256) {
    const int c = c0 + (q <= 256 ? (int)threadIdx.x % q : (int)threadIdx.x), grp = q <= 256 ? threadIdx.x / q : 0;
    Sum3 s[4];
    if (c < q && grp < groups) {
      unsigned seen = 0;
      for (size_t p = (size_t)blockIdx.x * groups + grp; p < pixels; p += (size_t)gridDim.x * groups) {
        const float4 v = *reinterpret_cast<const float4 *>(g + p * cp + c * 4);
        s[0].add(v.x); s[1].add(v.y); s[2].add(v.z); s[3].add(v.w);
        if ((++seen & 255u) == 0)
#pragma unroll
          for (int i = 0; i < 4; ++i) s[i].renorm();
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) sd[threadIdx.x][i] = s[i];
    __syncthreads();
    add_groups(sd, min(q, 256), groups);
    if ((int)threadIdx.x < min(q, 256) && c < q) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (c * 4 + i < C) partial[(size_t)blockIdx.x * C + c * 4 + i] = sd[threadIdx.x][i];
    }
  }
}

// x [B][3][plane] FP32 -> NHWC BF16 [pixel][16]: the high, middle and low parts
// of the 3 channels (the forward weights of all but the high ones are zero).
__global__ void pack_input(const float *__restrict__ x, bf16 *__restrict__ y, int B, size_t plane) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)B * plane;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t b = i / plane, p = i - b * plane;
    const float *s = x + b * 3 * plane + p;
    const float v[3] = {s[0], s[plane], s[2 * plane]};
    bf16 o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) o[c] = __float2bfloat16(0.f);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const bf16 h = __float2bfloat16(v[c]);
      // no rest beside an infinite high part: its NaN times the zero weights would hide it
      const float r = isinf(__bfloat162float(h)) ? 0.f : v[c] - __bfloat162float(h);
      const bf16 m = __float2bfloat16(r);
      o[c] = h;
      o[3 + c] = m;
      o[6 + c] = __float2bfloat16(r - __bfloat162float(m));
    }
    uint4 *d = reinterpret_cast<uint4 *>(y + i * 16);
    d[0] = *reinterpret_cast<const uint4 *>(o);
    d[1] = *reinterpret_cast<const uint4 *>(o + 8);
  }
}

// 2 x 2 average pooling, 8 channels per thread (BF16 -> BF16); blockIdx.y =
// sample here and in the next two (32-bit indices within a sample).
__global__ void pool2_fwd(const bf16 *__restrict__ x, bf16 *__restrict__ y, int h, int w, int cp) {
  const unsigned q = cp / 8, n = (unsigned)h * w * q;
  const size_t b = blockIdx.y;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const unsigned c = i % q, p = i / q, xx = p % w, yy = p / w;
    const uint4 *s = reinterpret_cast<const uint4 *>(x) + (b * 4 * h * w + (size_t)(2 * yy) * (2 * w) + 2 * xx) * q + c;
    const uint4 v[4] = {s[0], s[q], s[(size_t)2 * w * q], s[(size_t)2 * w * q + q]};
    unsigned o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      unsigned u[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) u[j] = reinterpret_cast<const unsigned *>(&v[j])[k];
      const float a = bf16_lo(u[0]) + bf16_lo(u[1]) + bf16_lo(u[2]) + bf16_lo(u[3]);
      const float b = bf16_hi(u[0]) + bf16_hi(u[1]) + bf16_hi(u[2]) + bf16_hi(u[3]);
      o[k] = bf16_pack2(0.25f * a, 0.25f * b);
    }
    reinterpret_cast<uint4 *>(y)[b * n + i] = make_uint4(o[0], o[1], o[2], o[3]);
  }
}
// Its adjoint plus the skip gradient, under the ReLU mask of the pooled
// activation: gx = (gy / 4 + gskip) (act > 0); [B][2h][2w][cp], 4 channels per
// thread.
__global__ void pool2_bwd(const float *__restrict__ gy, const float *__restrict__ gskip, const bf16 *__restrict__ act,
                          float *__restrict__ gx, int h, int w, int cp) {
  const unsigned q = cp / 4, W = 2 * w, n = 2u * h * W * q;
  const size_t b = blockIdx.y;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const unsigned c = i % q, p = i / q, x = p % W, y = p / W;
    const float4 g = reinterpret_cast<const float4 *>(gy)[((b * h + (y >> 1)) * w + (x >> 1)) * q + c];
    const float4 k = reinterpret_cast<const float4 *>(gskip)[b * n + i];
    const uint2 a = reinterpret_cast<const uint2 *>(act)[b * n + i];
    float4 o;
    o.x = bf16_lo(a.x) > 0.f ? fmaf(0.25f, g.x, k.x) : 0.f;
    o.y = bf16_hi(a.x) > 0.f ? fmaf(0.25f, g.y, k.y) : 0.f;
    o.z = bf16_lo(a.y) > 0.f ? fmaf(0.25f, g.z, k.z) : 0.f;
    o.w = bf16_hi(a.y) > 0.f ? fmaf(0.25f, g.w, k.w) : 0.f;
    reinterpret_cast<float4 *>(gx)[b * n + i] = o;
  }
}
// Adjoint of the nearest 2x upsampling (2 x 2 sums) under the ReLU mask of the
// upsampled activation; output [B][h][w][cp].
__global__ void up2_bwd(const float *__restrict__ gy, const bf16 *__restrict__ act, float *__restrict__ gx, int h,
                        int w, int cp) {
  const unsigned q = cp / 4, n = (unsigned)h * w * q;
  const size_t b = blockIdx.y;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const unsigned c = i % q, p = i / q, x = p % w, y = p / w;
    const float4 *s = reinterpret_cast<const float4 *>(gy) + (b * 4 * h * w + (size_t)(2 * y) * (2 * w) + 2 * x) * q + c;
    const float4 v0 = s[0], v1 = s[q], v2 = s[(size_t)2 * w * q], v3 = s[(size_t)2 * w * q + q];
    const uint2 a = reinterpret_cast<const uint2 *>(act)[b * n + i];
    float4 o;
    o.x = bf16_lo(a.x) > 0.f ? v0.x + v1.x + v2.x + v3.x : 0.f;
    o.y = bf16_hi(a.x) > 0.f ? v0.y + v1.y + v2.y + v3.y : 0.f;
    o.z = bf16_lo(a.y) > 0.f ? v0.z + v1.z + v2.z + v3.z : 0.f;
    o.w = bf16_hi(a.y) > 0.f ? v0.w + v1.w + v2.w + v3.w : 0.f;
    reinterpret_cast<float4 *>(gx)[b * n + i] = o;
  }
}

// 1 x 1 head (C -> 1): y = sum_c w[c] a[c] + b, in channel order.
__global__ void head_fwd(const bf16 *__restrict__ a, const float *__restrict__ w, const float *__restrict__ bias,
                         float *__restrict__ y, size_t pixels, int C, int cp) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < pixels; i += (size_t)gridDim.x * blockDim.x) {
    const uint4 *s = reinterpret_cast<const uint4 *>(a + i * cp);
    float v = bias[0];
    for (int c = 0; c < C; c += 8) {
      const uint4 u = s[c >> 3];
      const unsigned k[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (c + j < C) v = fmaf(w[c + j], (j & 1) ? bf16_hi(k[j >> 1]) : bf16_lo(k[j >> 1]), v);
    }
    y[i] = v;
  }
}
// Head backward, one pass over the activation: gz[c] = w[c] gy under the ReLU mask
// of a, and per-block partials of the weight gradient sum_p a[c] gy and (slot C)
// of the bias gradient sum_p gy.  Threads as in channel_sums (4 channels each).
__global__ void __launch_bounds__(256) head_bwd(const float *__restrict__ gy, const bf16 *__restrict__ a,
                                                const float *__restrict__ w, float *__restrict__ gz, size_t pixels,
                                                int C, int cp, Sum3 *__restrict__ partial) {
  __shared__ Sum3 sd[256][5];
  const int q = cp / 4, groups = max(1, 256 / q);
  for (int c0 = 0; c0 < q; c0 += 256) {
    const int c = c0 + (q <= 256 ? (int)threadIdx.x % q : (int)threadIdx.x), grp = q <= 256 ? threadIdx.x / q : 0;
    Sum3 s[5];
    if (c < q && grp < groups) {
      float wv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) wv[i] = c * 4 + i < C ? w[c * 4 + i] : 0.f;
      unsigned seen = 0;
      for (size_t p = (size_t)blockIdx.x * groups + grp; p < pixels; p += (size_t)gridDim.x * groups) {
        const float gv = gy[p];
        const uint2 u = *reinterpret_cast<const uint2 *>(a + p * cp + c * 4);
        const float av[4] = {bf16_lo(u.x), bf16_hi(u.x), bf16_lo(u.y), bf16_hi(u.y)};
        float4 o;
        o.x = av[0] > 0.f ? wv[0] * gv : 0.f;
        o.y = av[1] > 0.f ? wv[1] * gv : 0.f;
        o.z = av[2] > 0.f ? wv[2] * gv : 0.f;
        o.w = av[3] > 0.f ? wv[3] * gv : 0.f;
        *reinterpret_cast<float4 *>(gz + p * cp + c * 4) = o;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float pr = av[i] * gv;
          s[i].add(pr);
          s[i].add(fmaf(av[i], gv, -pr));
        }
        s[4].add(gv);
        if ((++seen & 127u) == 0)
#pragma unroll
          for (int i = 0; i < 5; ++i) s[i].renorm();
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 5; ++i) sd[threadIdx.x][i] = s[i];
    __syncthreads();
    add_groups(sd, min(q, 256), groups);
    if ((int)threadIdx.x < min(q, 256) && c < q) {
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        const int slot = i < 4 ? c * 4 + i : C;
        if (i < 4 ? slot < C : c == 0) partial[(size_t)blockIdx.x * (C + 1) + slot] = sd[threadIdx.x][i];
      }
    }
  }
}

// Loss over n = B H W lattice values, d = y - t:
//   loss = (1/n) [ sum d^2 + lam sum_{lattice edges (p, q)} (d_p - d_q)^2 ]
// (lam = 0: mean squared error; the edge term is a discrete H1 seminorm, which
// weighs an error the way the operator's energy norm does: smooth errors
// little, pixel-scale noise much).  gy_p = (2/n) [d_p + lam sum_q (d_p - d_q)]
// over the lattice neighbours q of p.  Per-block partial sums of the loss.
__global__ void loss_kernel(const float *__restrict__ y, const float *__restrict__ t, float *__restrict__ gy,
                            int B, int H, int W, float lam, double *__restrict__ partial) {
  __shared__ double red[8];
  double s = 0.0;
  const size_t n = (size_t)B * H * W;
  const float sc = 2.0f / (float)n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    float g = d;
    double e = (double)d * d;
    if (lam != 0.f) {
      const int x = (int)(i % W), yy = (int)((i / W) % H);
      float lap = 0.f;
      if (x > 0) lap += d - (y[i - 1] - t[i - 1]);
      if (yy > 0) lap += d - (y[i - W] - t[i - W]);
      if (x + 1 < W) {
        const float dr = d - (y[i + 1] - t[i + 1]);
        lap += dr;
        e += (double)lam * dr * dr;
      }
      if (yy + 1 < H) {
        const float dd = d - (y[i + W] - t[i + W]);
        lap += dd;
        e += (double)lam * dd * dd;
      }
      g = fmaf(lam, lap, d);
    }
    gy[i] = sc * g;
    s += e;
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// FP32 weights of every 3 x 3 layer into its two packed BF16 copies (see
// Layouts); blockIdx.y = layer.
struct PackLayer {
  size_t woff, fwd, bwd;  // offsets into the parameters and the packed copies
  int cin, cout;
};
__global__ void pack_weights(const float *__restrict__ p, const PackLayer *__restrict__ ls, bf16 *__restrict__ out) {
  const PackLayer L = ls[blockIdx.y];
  const float *w = p + L.woff;
  const int nf = pad8(L.cout), nb = pad8(L.cin);
  const unsigned ef = (unsigned)chunks16(L.cin) * 9 * nf * 16, eb = (unsigned)chunks16(L.cout) * 9 * nb * 16;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < ef + eb; i += gridDim.x * blockDim.x) {
    const bool back = i >= ef;
    const unsigned e = back ? i - ef : i, n8 = back ? nb : nf;
    const int j = e & 15, n = (e >> 4) % n8, r = (e >> 4) / n8, tap = r % 9, k = (r / 9) * 16 + j;
    const int ci = back ? n : k, co = back ? k : n, tp = back ? 8 - tap : tap;
    const float v = ci < L.cin && co < L.cout ? w[((size_t)tp * L.cin + ci) * L.cout + co] : 0.f;
    out[(back ? L.bwd : L.fwd) + e] = __float2bfloat16(v);
  }
}

// Adam (FP32 master weights).
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, size_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float upd = lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = p[i] - upd;
  }
}

// ---------------------------------------------------------------------------
// Features and lift (solver side)
// ---------------------------------------------------------------------------
// s[m] = max |f_m| (one CTA per right-hand side)
__global__ void maxabs_kernel(const double *__restrict__ f, size_t n, double *__restrict__ s) {
  __shared__ double red[256];
  const double *p = f + (size_t)blockIdx.x * n;
  double v = 0.0;
  for (size_t i = threadIdx.x; i < n; i += blockDim.x) v = fmax(v, fabs(p[i]));
  red[threadIdx.x] = v;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
    __syncthreads();
  }
  if (threadIdx.x == 0) s[blockIdx.x] = red[0] > 0.0 ? red[0] : 1.0;
}

// x[m][0] = mean log kappa, x[m][1] = mean q, x[m][2] = mean f / s over the
// grid cells that fall into each lattice cell (area average when the grid is
// an integer multiple of the lattice, nearest sample otherwise).
__global__ void features_kernel(const double *__restrict__ kappa, const double *__restrict__ q,
                                const double *__restrict__ f, const double *__restrict__ s, int nr, int nz, int hw,
                                float *__restrict__ x) {
  const int m = blockIdx.y;
  const size_t plane = (size_t)hw * hw;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < plane; i += (size_t)gridDim.x * blockDim.x) {
    const int py = i / hw, px = i % hw;   // py along r, px along z
    const int fr = (nr % hw == 0) ? nr / hw : 1, fz = (nz % hw == 0) ? nz / hw : 1;
    const int r0 = (nr % hw == 0) ? py * fr : (int)(((long long)py * nr) / hw);
    const int z0 = (nz % hw == 0) ? px * fz : (int)(((long long)px * nz) / hw);
    double lk = 0.0, qq = 0.0, ff = 0.0;
    for (int a = 0; a < fr; ++a)
      for (int c = 0; c < fz; ++c) {
        const size_t e = (size_t)(r0 + a) * nz + z0 + c;
        lk += log(kappa[e]);
        qq += q[e];
        ff += f[(size_t)m * nr * nz + e];
      }
    const double inv = 1.0 / (fr * fz);
    x[((size_t)m * 3 + 0) * plane + i] = (float)(lk * inv);
    x[((size_t)m * 3 + 1) * plane + i] = (float)(qq * inv);
    x[((size_t)m * 3 + 2) * plane + i] = (float)(ff * inv / s[m]);
  }
}

// u[m][i][k] = s[m] * bilinear(y[m], at the lattice position of grid node (i, k)),
// lattice values sitting at cell centres ((p + 1/2) / hw).
// s[i] /= t for i < m (the feature scale of a lift whose training targets were
// u / s times t)
__global__ void div_scale_kernel(double *s, int m, double t) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) s[i] /= t;
}

__global__ void lift_kernel(const float *__restrict__ y, const double *__restrict__ s, int hw, int nr, int nz,
                            double *__restrict__ u) {
  const int m = blockIdx.y;
  const size_t n = (size_t)nr * nz;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int i = e / nz, k = e % nz;
    const float gy = ((i + 0.5f) * hw) / nr - 0.5f, gx = ((k + 0.5f) * hw) / nz - 0.5f;
    const int y0 = max(0, min(hw - 1, (int)floorf(gy))), x0 = max(0, min(hw - 1, (int)floorf(gx)));
    const int y1 = min(hw - 1, y0 + 1), x1 = min(hw - 1, x0 + 1);
    const float wy = fminf(fmaxf(gy - y0, 0.f), 1.f), wx = fminf(fmaxf(gx - x0, 0.f), 1.f);
    const float *p = y + (size_t)m * hw * hw;
    const float v = (1 - wy) * ((1 - wx) * p[y0 * hw + x0] + wx * p[y0 * hw + x1]) +
                    wy * ((1 - wx) * p[y1 * hw + x0] + wx * p[y1 * hw + x1]);
    u[(size_t)m * n + e] = s[m] * (double)v;
  }
}

int grid1d(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 4096); }

// ---------------------------------------------------------------------------
// Network object
// ---------------------------------------------------------------------------
struct NetLayer {
  char kind;     // 'c' conv+relu, 's' conv+relu+skip, 'p' pool, 'u' up, 'h' head
  int cin = 0, cout = 0, res = 0;  // res: spatial size of this layer's output
  size_t woff = 0, boff = 0;       // offsets into the flat parameter vector
  size_t fwd = 0, bwd = 0;         // offsets of the packed weights
  int in = -1, up = 0;             // input activation buffer (-1: the network's input), read 2x upsampled if up
  int out = -1, out2 = -1;         // activation buffers (out2: relu output + skip)
  int skip = -1;                   // buffer added after ReLU ('s')
};

struct GuessNet {
  int hw = 0, cap = 0;   // lattice size, batch capacity
  int ch[4] = {24, 48, 96, 192};
  std::vector<NetLayer> layers;
  size_t nparams = 0, npacked = 0;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // FP32 master, grads, Adam moments
  bf16 *pk = nullptr;                                            // packed BF16 weights
  PackLayer *pl = nullptr;                                       // device: the conv layers' packing
  int npack = 0;
  bf16 *xin = nullptr;                                           // packed input [cap][hw][hw][16]
  std::vector<std::pair<int, int>> bufshape;                     // (channels, res) per activation buffer
  std::vector<bf16 *> act;                                       // activations [cap][res][res][pad8(C)]
  float *y = nullptr, *gy = nullptr;                             // head output and its gradient [cap][hw][hw]
  float *gbuf[3] = {nullptr, nullptr, nullptr};                  // gradients (largest activation)
  std::vector<float *> gskip;                                    // skip gradients per level
  float *partial = nullptr;                                      // weight-gradient partials
  Sum3 *spart = nullptr;                                         // partials of the bias and head gradients
  double *lpart = nullptr;                                       // loss partials
  float h1 = 0.f;                                                // weight of the loss's edge term
  int step = 0;
};

size_t act_elems(const GuessNet *n, int buf) {
  return (size_t)n->cap * pad8(n->bufshape[buf].first) * n->bufshape[buf].second * n->bufshape[buf].second;
}

void build_layers(GuessNet *n) {
  const int c1 = n->ch[0], c2 = n->ch[1], c3 = n->ch[2], c4 = n->ch[3];
  const int H = n->hw;
  auto buf = [&](int c, int r) {
    n->bufshape.push_back({c, r});
    return (int)n->bufshape.size() - 1;
  };
  size_t off = 0, pack = 0;
  int cur = -1, up2 = 0;
  auto conv = [&](char kind, int cin, int cout, int res, int skip) {
    NetLayer L;
    L.kind = kind;
    L.in = cur;
    L.up = up2;
    up2 = 0;
    L.fwd = pack;
    pack += (size_t)chunks16(cin) * 9 * pad8(cout) * 16;
    L.bwd = pack;
    pack += (size_t)chunks16(cout) * 9 * pad8(cin) * 16;
    L.cin = cin;
    L.cout = cout;
    L.res = res;
    L.woff = off;
    off += (size_t)9 * cin * cout;
    L.boff = off;
    off += cout;
    L.out = buf(cout, res);
    if (kind == 's') {
      L.out2 = buf(cout, res);
      L.skip = skip;
    }
    n->layers.push_back(L);
    return cur = (kind == 's') ? L.out2 : L.out;
  };
  auto pool = [&](int c, int res) {
    NetLayer L;
    L.kind = 'p';
    L.cin = L.cout = c;
    L.res = res;
    L.in = cur;
    L.out = cur = buf(c, res);
    n->layers.push_back(L);
    return L.out;
  };
  auto up = [&](int c, int res) {
    NetLayer L;
    L.kind = 'u';  // read upsampled by the next convolution: no buffer of its own
    L.cin = L.cout = c;
    L.res = res;
    L.in = L.out = cur;
    up2 = 1;
    n->layers.push_back(L);
  };
  conv('c', 3, c1, H, -1);
  const int s1 = conv('c', c1, c1, H, -1);
  pool(c1, H / 2);
  conv('c', c1, c2, H / 2, -1);
  const int s2 = conv('c', c2, c2, H / 2, -1);
  pool(c2, H / 4);
  conv('c', c2, c3, H / 4, -1);
  const int s3 = conv('c', c3, c3, H / 4, -1);
  pool(c3, H / 8);
  conv('c', c3, c4, H / 8, -1);
  conv('c', c4, c4, H / 8, -1);
  up(c4, H / 4);
  conv('s', c4, c3, H / 4, s3);
  conv('c', c3, c3, H / 4, -1);
  up(c3, H / 2);
  conv('s', c3, c2, H / 2, s2);
  conv('c', c2, c2, H / 2, -1);
  up(c2, H);
  conv('s', c2, c1, H, s1);
  conv('c', c1, c1, H, -1);
  NetLayer hd;
  hd.kind = 'h';
  hd.cin = c1;
  hd.cout = 1;
  hd.res = H;
  hd.in = cur;
  hd.woff = off;
  off += c1;
  hd.boff = off;
  off += 1;
  n->layers.push_back(hd);
  n->nparams = off;
  n->npacked = pack;
}

// deterministic host initialisation: He-normal weights (Box-Muller on a
// splitmix64 stream), zero biases
uint64_t splitmix64(uint64_t &x) {
  uint64_t z = (x += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
double uniform01(uint64_t &st) { return ((splitmix64(st) >> 11) + 0.5) * (1.0 / 9007199254740992.0); }

void init_host_params(const GuessNet *n, uint64_t seed, std::vector<float> &h) {
  h.assign(n->nparams, 0.f);
  uint64_t st = seed;
  for (const NetLayer &L : n->layers) {
    if (L.kind == 'p' || L.kind == 'u') continue;
    const size_t nw = (L.kind == 'h') ? (size_t)L.cin : (size_t)9 * L.cin * L.cout;
    const double fan_in = (L.kind == 'h') ? L.cin : 9.0 * L.cin;
    const double sd = (L.kind == 'h') ? std::sqrt(1.0 / fan_in) : std::sqrt(2.0 / fan_in);
    for (size_t i = 0; i < nw; ++i) {
      const double u1 = uniform01(st), u2 = uniform01(st);
      h[L.woff + i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(2.0 * M_PI * u2));
    }
  }
}

template <typename P>
cudaError_t zalloc(P **p, size_t count) {
  *p = nullptr;
  if (count == 0) return cudaSuccess;
  cudaError_t e = cudaMalloc((void **)p, count * sizeof(P));
  // the fill runs on the legacy stream: finish it before any launch on a
  // non-blocking stream can touch the buffer
  if (e == cudaSuccess) e = cudaMemset(*p, 0, count * sizeof(P));
  if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
  return e;
}

void net_free(GuessNet *n) {
  cudaFree(n->p); cudaFree(n->g); cudaFree(n->m); cudaFree(n->v); cudaFree(n->pk); cudaFree(n->pl);
  cudaFree(n->xin); cudaFree(n->gy);
  for (auto *a : n->act) cudaFree(a);
  for (auto *a : n->gskip) cudaFree(a);
  cudaFree(n->y);
  for (float *g : n->gbuf) cudaFree(g);
  cudaFree(n->partial); cudaFree(n->spart); cudaFree(n->lpart);
  delete n;
}

// ---------------------------------------------------------------------------
// passes
// ---------------------------------------------------------------------------
// Columns of 8 output channels per CTA: 6 where that divides their number, else
// 3; rows of pixels per warp: 2, or 1 where the grid would not cover the SMs
// twice.
template <int NT, int MW, int PLANES>
void launch_conv_shape(const ConvArgs &a, int B, cudaStream_t s) {
  using S = ConvShape<NT, MW, PLANES>;
  ensure_smem_attr((const void *)conv3x3_kernel<NT, MW, PLANES>, S::smem);
  const dim3 grid(((a.W + 15) / 16) * ((a.H + 8 * MW - 1) / (8 * MW)), (pad8(a.cout) / 8 + NT - 1) / NT, B);
  note_launch();
  conv3x3_kernel<NT, MW, PLANES><<<grid, 256, S::smem, s>>>(a);
}
template <int PLANES>
void launch_conv(const ConvArgs &a, int B, cudaStream_t s) {
  const int nt = pad8(a.cout) / 8;
  const bool wide = PLANES == 1 && nt % 6 == 0;
  const long long ctas = (long long)((a.W + 15) / 16) * ((a.H + 15) / 16) * B * ((nt + 2) / 3) / (wide ? 2 : 1);
  const bool tall = ctas >= 304;
  if (PLANES == 1 && wide) {
    if (tall) launch_conv_shape<6, 2, 1>(a, B, s);
    else launch_conv_shape<6, 1, 1>(a, B, s);
  } else {
    // three planes: twice the columns of one row per warp where they divide (an
    // input patch is split anew for every column block)
    if (PLANES == 3 && nt % 6 == 0) launch_conv_shape<6, 1, PLANES>(a, B, s);
    else if (tall) launch_conv_shape<3, 2, PLANES>(a, B, s);
    else launch_conv_shape<3, 1, PLANES>(a, B, s);
  }
}

constexpr int kWgCtas = 304;    // weight-gradient CTAs in all: two rounds of 152 SMs
constexpr int kSumBlocks = 912; // blocks of the channel sums
int wgrad_splits(int cin, int cout, long long tiles) {
  const int blocks = chunks16(cin) * ((cout + kWgN - 1) / kWgN);
  return (int)std::max<long long>(1, std::min<long long>(tiles, kWgCtas / blocks));
}

// Writes dW [9][cin][cout].  planes = 3: the network's input (see
// pack_input), cin = 3.
void launch_wgrad(GuessNet *n, const bf16 *in, const float *gz, float *gw, int B, int cin, int cout, int res, int up,
                  int planes, cudaStream_t s) {
  const int vcin = planes == 3 ? 9 : cin;
  WgradArgs a{in, gz, n->partial, vcin, planes == 3 ? 16 : pad8(cin), cout, B, res, res, up};
  const int tiles1 = (res + 15) / 16;
  const int splits = wgrad_splits(vcin, cout, (long long)B * tiles1 * tiles1);
  ensure_smem_attr((const void *)conv3x3_wgrad_kernel, kWgSmem);
  note_launch();
  conv3x3_wgrad_kernel<<<dim3(chunks16(vcin), (cout + kWgN - 1) / kWgN, splits), 256, kWgSmem, s>>>(a);
  const size_t nw = (size_t)9 * cin * cout;
  note_launch();
  sum_partials<<<(unsigned)((nw + 31) / 32), 256, 0, s>>>(n->partial, splits, nw, gw, planes, cout);
}

void bias_grad(GuessNet *n, const float *gz, float *gb, int B, int C, int res, cudaStream_t s) {
  note_launch();
  channel_sums<<<kSumBlocks, 256, 0, s>>>(gz, C, pad8(C), (size_t)B * res * res, n->spart);
  note_launch();
  sum_sum3<<<(C + 7) / 8, 256, 0, s>>>(n->spart, kSumBlocks, C, gb);
}

void pack_all(GuessNet *n, cudaStream_t s) {
  note_launch();
  pack_weights<<<dim3(152, n->npack), 256, 0, s>>>(n->p, n->pl, n->pk);
}

void forward_pass(GuessNet *n, const float *x, int B, cudaStream_t s) {
  const int H = n->hw;
  note_launch();
  pack_input<<<grid1d((size_t)B * H * H), 256, 0, s>>>(x, n->xin, B, (size_t)H * H);
  for (const NetLayer &L : n->layers) {
    if (L.kind == 'c' || L.kind == 's') {
      // the packed input has 16 channels, of which the weights use the first 3
      const bool first = L.in < 0;
      ConvArgs a{first ? n->xin : n->act[L.in], n->pk + L.fwd, n->p + L.boff, n->act[L.out],
                 L.kind == 's' ? n->act[L.out2] : nullptr, L.kind == 's' ? n->act[L.skip] : nullptr, nullptr,
                 first ? 16 : L.cin, L.cout, L.res, L.res, L.up};
      launch_conv<1>(a, B, s);
    } else if (L.kind == 'p') {
      note_launch();
      pool2_fwd<<<dim3(grid1d((size_t)L.res * L.res * pad8(L.cout) / 8), B), 256, 0, s>>>(
          n->act[L.in], n->act[L.out], L.res, L.res, pad8(L.cout));
    } else if (L.kind == 'h') {
      note_launch();
      head_fwd<<<grid1d((size_t)B * H * H), 256, 0, s>>>(n->act[L.in], n->p + L.woff, n->p + L.boff, n->y,
                                                         (size_t)B * H * H, L.cin, pad8(L.cin));
    }
  }
}

// Backward pass from n->gy (d loss / d y, FP32 [B][H][W]); fills n->g.  Every
// gradient buffer that a weight gradient reads already carries the ReLU mask of
// its activation (written so by the kernel that forms it).
void backward_pass(GuessNet *n, int B, cudaStream_t s) {
  const int H = n->hw, last = (int)n->layers.size() - 1;
  float *g = n->gbuf[0], *other = n->gbuf[1], *high = n->gbuf[2];
  std::vector<float *> skips;
  {
    const NetLayer &L = n->layers[last];
    note_launch();
    head_bwd<<<kSumBlocks, 256, 0, s>>>(n->gy, n->act[L.in], n->p + L.woff, g, (size_t)B * H * H, L.cin, pad8(L.cin),
                                        n->spart);
    note_launch();
    sum_sum3<<<(L.cin + 8) / 8, 256, 0, s>>>(n->spart, kSumBlocks, L.cin + 1, n->g + L.woff);
  }
  for (int li = last - 1; li >= 0; --li) {
    const NetLayer &L = n->layers[li];
    if (L.kind != 'c' && L.kind != 's') continue;  // 'p', 'u': with the convolution behind them
    const bool first = L.in < 0;
    launch_wgrad(n, first ? n->xin : n->act[L.in], g, n->g + L.woff, B, L.cin, L.cout, L.res, L.up, first ? 3 : 1, s);
    bias_grad(n, g, n->g + L.boff, B, L.cout, L.res, s);
    if (li == 0) break;
    const NetLayer &prev = n->layers[li - 1];
    ConvArgs a{g, n->pk + L.bwd, nullptr, other, nullptr, nullptr, nullptr, L.cout, L.cin, L.res, L.res, 0};
    if (prev.kind == 'c') {
      a.mask = n->act[prev.out];
    } else if (prev.kind == 's') {  // the skip source receives the gradient unmasked
      float *sg = n->gskip[skips.size()];
      skips.push_back(sg);
      a.out2 = sg;
      a.mask = n->act[prev.out];
    } else {
      a.out = high;
    }
    launch_conv<3>(a, B, s);
    if (prev.kind == 'p') {
      float *sg = skips.back();
      skips.pop_back();
      note_launch();
      pool2_bwd<<<dim3(grid1d((size_t)4 * L.res * L.res * pad8(L.cin) / 4), B), 256, 0, s>>>(
          high, sg, n->act[prev.in], other, L.res, L.res, pad8(L.cin));
    } else if (prev.kind == 'u') {
      // masked by the ReLU of the convolution whose output is upsampled
      note_launch();
      up2_bwd<<<dim3(grid1d((size_t)(L.res / 2) * (L.res / 2) * pad8(L.cin) / 4), B), 256, 0, s>>>(
          high, n->act[n->layers[li - 2].out], other, L.res / 2, L.res / 2, pad8(L.cin));
    }
    std::swap(g, other);
  }
}

int loss_and_grad(GuessNet *n, const float *target, int B, cudaStream_t s, double *loss) {
  const size_t N = (size_t)B * n->hw * n->hw;
  const int blocks = std::min<int>(grid1d(N), 1024);
  note_launch();
  loss_kernel<<<blocks, 256, 0, s>>>(n->y, target, n->gy, B, n->hw, n->hw, n->h1, n->lpart);
  std::vector<double> h(blocks);
  if (cudaMemcpyAsync(h.data(), n->lpart, blocks * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return AX_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return AX_ERR_CUDA;
  double sum = 0.0;
  for (double v : h) sum += v;
  if (loss) *loss = sum / N;
  return AX_OK;
}

}  // namespace
}  // namespace ax

using namespace ax;

extern "C" {

int ax_guessnet_create(int32_t hw, const int32_t *channels, int32_t batch_capacity, uint64_t seed, void **out) {
  if (!out) return AX_ERR_INVALID_ARG;
  *out = nullptr;
  if (hw < 8 || hw % 8 != 0 || hw > 4096 || batch_capacity < 1) return AX_ERR_INVALID_ARG;
  GuessNet *n = new GuessNet();
  n->hw = hw;
  n->cap = batch_capacity;
  if (channels)
    for (int i = 0; i < 4; ++i) {
      if (channels[i] < 1 || channels[i] > 1024) {
        delete n;
        return AX_ERR_INVALID_ARG;
      }
      n->ch[i] = channels[i];
    }
  build_layers(n);
  std::vector<float> h;
  init_host_params(n, seed, h);
  cudaError_t e = zalloc(&n->p, n->nparams);
  if (e == cudaSuccess) e = zalloc(&n->g, n->nparams);
  if (e == cudaSuccess) e = zalloc(&n->m, n->nparams);
  if (e == cudaSuccess) e = zalloc(&n->v, n->nparams);
  if (e == cudaSuccess) e = zalloc(&n->pk, n->npacked);
  if (e == cudaSuccess) e = zalloc(&n->xin, (size_t)batch_capacity * hw * hw * 16);
  std::vector<PackLayer> pls;
  for (const NetLayer &L : n->layers)
    if (L.kind == 'c' || L.kind == 's') pls.push_back({L.woff, L.fwd, L.bwd, L.cin, L.cout});
  n->npack = (int)pls.size();
  if (e == cudaSuccess) e = zalloc(&n->pl, pls.size());
  if (e == cudaSuccess) e = cudaMemcpy(n->pl, pls.data(), pls.size() * sizeof(PackLayer), cudaMemcpyHostToDevice);
  size_t maxact = 0;
  for (size_t b = 0; b < n->bufshape.size() && e == cudaSuccess; ++b) {
    bf16 *a = nullptr;
    e = zalloc(&a, act_elems(n, (int)b));
    n->act.push_back(a);
    maxact = std::max(maxact, act_elems(n, (int)b));
  }
  // a gradient of an upsampled activation has 4 times its pixels
  for (const NetLayer &L : n->layers)
    if (L.up) maxact = std::max(maxact, (size_t)n->cap * pad8(L.cin) * L.res * L.res);
  if (e == cudaSuccess) e = zalloc(&n->y, (size_t)n->cap * hw * hw);
  if (e == cudaSuccess) e = zalloc(&n->gy, (size_t)n->cap * hw * hw);
  for (float *&g : n->gbuf)
    if (e == cudaSuccess) e = zalloc(&g, maxact);
  for (int k = 0; k < 3 && e == cudaSuccess; ++k) {
    float *sg = nullptr;
    e = zalloc(&sg, maxact);
    n->gskip.push_back(sg);
  }
  // partials of the weight gradients (splits x 9 cin cout) and of the channel sums
  size_t pn = 0, sn = 0;
  for (const NetLayer &L : n->layers) {
    const int cin = L.in < 0 ? 9 : L.cin;
    if (L.kind == 'c' || L.kind == 's')
      pn = std::max(pn, (size_t)wgrad_splits(cin, L.cout, 1LL << 40) * 9 * cin * L.cout);
    sn = std::max(sn, (size_t)kSumBlocks * (std::max(L.cin, L.cout) + 1));
  }
  if (e == cudaSuccess) e = zalloc(&n->partial, pn);
  if (e == cudaSuccess) e = zalloc(&n->spart, sn);
  if (e == cudaSuccess) e = zalloc(&n->lpart, 1024);
  if (e == cudaSuccess) e = cudaMemcpy(n->p, h.data(), n->nparams * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    pack_all(n, nullptr);
    e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    net_free(n);
    return e == cudaErrorMemoryAllocation ? AX_ERR_OOM : AX_ERR_CUDA;
  }
  *out = n;
  return AX_OK;
}

int ax_guessnet_destroy(void *net) {
  if (net) net_free((GuessNet *)net);
  return AX_OK;
}

int64_t ax_guessnet_num_params(void *net) { return net ? (int64_t)((GuessNet *)net)->nparams : 0; }

int ax_guessnet_get_params(void *net, float *host, int64_t n) {
  GuessNet *g = (GuessNet *)net;
  if (!g || !host || n != (int64_t)g->nparams) return AX_ERR_INVALID_ARG;
  return cudaMemcpy(host, g->p, n * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? AX_OK : AX_ERR_CUDA;
}

int ax_guessnet_set_params(void *net, const float *host, int64_t n) {
  GuessNet *g = (GuessNet *)net;
  if (!g || !host || n != (int64_t)g->nparams) return AX_ERR_INVALID_ARG;
  if (cudaMemcpy(g->p, host, n * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return AX_ERR_CUDA;
  pack_all(g, nullptr);
  cudaMemset(g->m, 0, n * sizeof(float));
  cudaMemset(g->v, 0, n * sizeof(float));
  g->step = 0;
  return cudaDeviceSynchronize() == cudaSuccess ? AX_OK : AX_ERR_CUDA;
}

int ax_guessnet_forward(void *net, const float *x, float *y, int32_t batch, void *stream) {
  GuessNet *n = (GuessNet *)net;
  if (!n || !x || !y || batch < 1 || batch > n->cap) return AX_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  forward_pass(n, x, batch, s);
  cudaMemcpyAsync(y, n->y, (size_t)batch * n->hw * n->hw * sizeof(float), cudaMemcpyDeviceToDevice, s);
  return cudaGetLastError() == cudaSuccess ? AX_OK : AX_ERR_CUDA;
}

int ax_guessnet_set_loss(void *net, double h1_weight) {
  GuessNet *g = (GuessNet *)net;
  if (!g || !(h1_weight >= 0.0) || h1_weight > 1e6) return AX_ERR_INVALID_ARG;
  g->h1 = (float)h1_weight;
  return AX_OK;
}

int ax_guessnet_gradients(void *net, const float *x, const float *target, int32_t batch, float *grad_host,
                          double *loss, void *stream) {
  GuessNet *n = (GuessNet *)net;
  if (!n || !x || !target || batch < 1 || batch > n->cap) return AX_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  forward_pass(n, x, batch, s);
  int rc = loss_and_grad(n, target, batch, s, loss);
  if (rc != AX_OK) return rc;
  backward_pass(n, batch, s);
  if (grad_host) {
    if (cudaMemcpyAsync(grad_host, n->g, n->nparams * sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess)
      return AX_ERR_CUDA;
  }
  return cudaStreamSynchronize(s) == cudaSuccess ? AX_OK : AX_ERR_CUDA;
}

int ax_guessnet_train_step(void *net, const float *x, const float *target, int32_t batch, float lr, double *loss,
                           void *stream) {
  GuessNet *n = (GuessNet *)net;
  if (!n || !(lr > 0.f)) return AX_ERR_INVALID_ARG;
  int rc = ax_guessnet_gradients(net, x, target, batch, nullptr, loss, stream);
  if (rc != AX_OK) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  n->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)n->step), c2 = 1.f - std::pow(b2, (float)n->step);
  note_launch();
  adam_kernel<<<grid1d(n->nparams), 256, 0, s>>>(n->p, n->g, n->m, n->v, n->nparams, lr, b1, b2, 1e-8f, c1, c2);
  pack_all(n, s);
  return cudaGetLastError() == cudaSuccess ? AX_OK : AX_ERR_CUDA;
}

int ax_guessnet_save(void *net, const char *path) {
  GuessNet *n = (GuessNet *)net;
  if (!n || !path) return AX_ERR_INVALID_ARG;
  std::vector<float> h(n->nparams);
  if (cudaMemcpy(h.data(), n->p, h.size() * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return AX_ERR_CUDA;
  FILE *fp = fopen(path, "wb");
  if (!fp) return AX_ERR_INVALID_ARG;
  // header: magic, version, hw, channels[4], nparams; then FP32 little-endian
  // parameters and a 64-bit FNV-1a checksum of their bytes
  const int32_t hdr[8] = {0x4e475841 /* "AXGN" */, 1, n->hw, n->ch[0], n->ch[1], n->ch[2], n->ch[3],
                          (int32_t)n->nparams};
  uint64_t sum = 1469598103934665603ull;
  const unsigned char *bytes = reinterpret_cast<const unsigned char *>(h.data());
  for (size_t i = 0; i < h.size() * sizeof(float); ++i) sum = (sum ^ bytes[i]) * 1099511628211ull;
  const bool ok = fwrite(hdr, sizeof(hdr), 1, fp) == 1 && fwrite(h.data(), sizeof(float), h.size(), fp) == h.size() &&
                  fwrite(&sum, sizeof(sum), 1, fp) == 1;
  fclose(fp);
  return ok ? AX_OK : AX_ERR_INVALID_ARG;
}

int ax_guessnet_load(void *net, const char *path) {
  GuessNet *n = (GuessNet *)net;
  if (!n || !path) return AX_ERR_INVALID_ARG;
  FILE *fp = fopen(path, "rb");
  if (!fp) return AX_ERR_INVALID_ARG;
  int32_t hdr[8];
  std::vector<float> h(n->nparams);
  uint64_t sum = 0;
  bool ok = fread(hdr, sizeof(hdr), 1, fp) == 1 && hdr[0] == 0x4e475841 && hdr[1] == 1 && hdr[2] == n->hw &&
            hdr[3] == n->ch[0] && hdr[4] == n->ch[1] && hdr[5] == n->ch[2] && hdr[6] == n->ch[3] &&
            hdr[7] == (int32_t)n->nparams && fread(h.data(), sizeof(float), h.size(), fp) == h.size() &&
            fread(&sum, sizeof(sum), 1, fp) == 1;
  fclose(fp);
  if (!ok) return AX_ERR_INVALID_ARG;
  uint64_t chk = 1469598103934665603ull;
  const unsigned char *bytes = reinterpret_cast<const unsigned char *>(h.data());
  for (size_t i = 0; i < h.size() * sizeof(float); ++i) chk = (chk ^ bytes[i]) * 1099511628211ull;
  if (chk != sum) return AX_ERR_INVALID_ARG;
  return ax_guessnet_set_params(net, h.data(), (int64_t)h.size());
}

int ax_guessnet_features(const double *kappa, const double *q, const double *f, int32_t m, int32_t nr, int32_t nz,
                         int32_t hw, float *x, double *scale, void *stream) {
  if (!kappa || !q || !f || !x || !scale || m < 1 || nr < 1 || nz < 1 || hw < 1) return AX_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  note_launch();
  maxabs_kernel<<<m, 256, 0, s>>>(f, (size_t)nr * nz, scale);
  note_launch();
  features_kernel<<<dim3(grid1d((size_t)hw * hw), m), 256, 0, s>>>(kappa, q, f, scale, nr, nz, hw, x);
  return cudaGetLastError() == cudaSuccess ? AX_OK : AX_ERR_CUDA;
}

int ax_guessnet_lift(const float *y, int32_t m, int32_t hw, const double *scale, int32_t nr, int32_t nz, double *u,
                     void *stream) {
  if (!y || !scale || !u || m < 1 || nr < 1 || nz < 1 || hw < 1) return AX_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  note_launch();
  lift_kernel<<<dim3(grid1d((size_t)nr * nz), m), 256, 0, s>>>(y, scale, hw, nr, nz, u);
  return cudaGetLastError() == cudaSuccess ? AX_OK : AX_ERR_CUDA;
}

int ax_solve_learned(ax_operator *op, void *net, const double *kappa, const double *q, const double *f, double *u,
                     int32_t m, double tol, int32_t max_iter, int32_t method, int32_t flags, int32_t pre,
                     double target_scale, ax_solve_info *info, void *stream) {
  GuessNet *n = (GuessNet *)net;
  if (!op || !n || !kappa || !q || !f || !u || m < 1 || !(target_scale > 0.0) || !std::isfinite(target_scale))
    return AX_ERR_INVALID_ARG;
  if (flags & AX_FLAG_HOST_BUFFERS) return AX_ERR_UNSUPPORTED;
  const int32_t nr = op->nr, nz = op->nz;
  cudaStream_t s = (cudaStream_t)stream;
  const int hw = n->hw;
  float *x = nullptr, *y = nullptr;
  double *sc = nullptr;
  struct Free {
    float *x, *y;
    double *sc;
    ~Free() {
      if (x) cudaFree(x);
      if (y) cudaFree(y);
      if (sc) cudaFree(sc);
    }
  } hold{nullptr, nullptr, nullptr};
  if (cudaMalloc(&x, (size_t)m * 3 * hw * hw * sizeof(float)) != cudaSuccess) return AX_ERR_OOM;
  hold.x = x;
  if (cudaMalloc(&y, (size_t)m * hw * hw * sizeof(float)) != cudaSuccess) return AX_ERR_OOM;
  hold.y = y;
  if (cudaMalloc(&sc, (size_t)m * sizeof(double)) != cudaSuccess) return AX_ERR_OOM;
  hold.sc = sc;
  int rc = pre ? ax_guessnet_features_pre(op, kappa, q, f, m, hw, x, sc, stream)
               : ax_guessnet_features(kappa, q, f, m, nr, nz, hw, x, sc, stream);
  if (rc != AX_OK) return rc;
  for (int c = 0; c < m; c += n->cap) {  // the network's batches
    const int b = std::min(n->cap, m - c);
    if ((rc = ax_guessnet_forward(net, x + (size_t)c * 3 * hw * hw, y + (size_t)c * hw * hw, b, stream)) != AX_OK)
      return rc;
  }
  if (target_scale != 1.0) {
    note_launch();
    div_scale_kernel<<<(m + 255) / 256, 256, 0, s>>>(sc, m, target_scale);
  }
  if ((rc = ax_guessnet_lift(y, m, hw, sc, nr, nz, u, stream)) != AX_OK) return rc;
  return ax_solve(op, f, u, m, tol, max_iter, method, flags | AX_FLAG_USE_GUESS | AX_FLAG_CHECK_GUESS, info,
                  stream);
}

}  // extern "C"
