// Variable-coefficient cylindrical 5-point stencil (Section 2.1, Eqs.
// poisson_diff_2, scheme_op_r_z, diff_approx1, sign-reversed so A > 0):
//
//   (A y)_{i,k} = CR_i (y_{i,k} - y_{i+1,k}) + CR_{i-1} (y_{i,k} - y_{i-1,k})
//               + CZ_{i,k} (y_{i,k} - y_{i,k+1}) + CZ_{i,k-1} (y_{i,k} - y_{i,k-1})
//               + W_{i,k} y_{i,k}
//
// with CR = KR / h_r^2, CZ = KZ / h_z^2 precomputed, CR_0 = 0 on the axis and
// zero values beyond the Dirichlet boundaries r = lr, z = 0, z = lz.
//
// A warp owns 2 consecutive r-rows and a strip of 32 short vectors (4 FP32 / 2
// FP64) of consecutive z-nodes; z-neighbours across lanes come from warp
// shuffles, and the two warp-edge lanes fetch one extra element.
#include <algorithm>
#include "ax_finish.cuh"

namespace ax {

namespace {

template <typename T, int MODE>
struct StencilValue {
  // Value of the grid function the operator is applied to, at element e.
  __device__ __forceinline__ static T at(const T *in, const T *p_old, size_t e, T beta) {
    if (MODE == kStencilPcg && beta != T(0)) return in[e] + beta * p_old[e];  // p_1 = z
    return in[e];
  }
};

// Hint: bring the line holding p into L2 (no register, no completion; p must
// be a valid global address).
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

constexpr int kRowsLong = 16;  // rows per CTA of stencil_kernel, at most
constexpr int kStripRows = 2;  // rows per warp of strip_kernel
constexpr int kStripChunk = 8; // right-hand sides per CTA of strip_kernel, at most

// 4-, 8- or 16-byte asynchronous global -> shared copies, zero fill when !ok.
template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src, bool ok) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES),
                 "r"(ok ? BYTES : 0)
                 : "memory");
}

// 2 rows per warp and a loop over up to 8 right-hand sides, with the
// coefficients of the strip kept in registers (12 B per node, read from L2 once
// per 8 right-hand sides) and the rows of the next ones copied asynchronously
// into a ring of shared-memory stages of the warp's own.  What bounds the pass
// is memory latency: a register window walked down 16 rows (below) has one row
// of loads per warp in flight and waits one round trip per row; here each warp
// has the 2 KB stages of 3 right-hand sides in flight and waits for no other
// warp.
// Warps per CTA depend on the grid only (strip_warps), and a CTA's partial is
// formed for each right-hand side from the same nodes in the same order however
// many share the launch, so results do not depend on that.
template <typename T, int MODE>
struct StripShape {
  static constexpr int V = VecT<T>::n;
  static constexpr int arrays = MODE == kStencilPcg ? 2 : 1;  // z and p_old, or the grid function
  static constexpr int stages = MODE == kStencilPcg ? 3 : 4;
  static constexpr int row = 32 * V;                          // elements of a strip row
  static constexpr int array = (kStripRows + 2) * row + 16 / (int)sizeof(T) * kStripRows;  // rows, then edges
  static constexpr int stage = arrays * array;
  // a warp's ring: no more stages than right-hand sides (few: more CTAs fit an SM.
  // Mixed solves, all stages and these, four alternating runs of each within 0.2%: one
  // 1024 x 1024 2.087 and 2.068 ms, three 4.273 and 4.233, one 1500 x 1500 5.056 and
  // 4.994; 700 x 700 to 3000 x 3000 the same)
  __host__ __device__ static size_t warp_bytes(int chunk) {
    return (size_t)(chunk < stages ? chunk : stages) * stage * sizeof(T);
  }
};

template <typename T, int MODE, int NW>
__global__ void __launch_bounds__(32 * NW, (MODE == kStencilPcg ? 16 : 24) / NW)
    strip_kernel(const StencilArgs<T> a, int chunk) {
  using S = StripShape<T, MODE>;
  constexpr int V = S::V, R = kStripRows;
  extern __shared__ __align__(16) unsigned char ssm[];
  __shared__ T s_acc[kStripChunk][32 * NW];
  __shared__ double red[NW];
  __shared__ int s_m[kStripChunk], s_odd[kStripChunk], s_last[kStripChunk], s_n;
  __shared__ T s_beta[kStripChunk];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nr = a.nr, nz = a.nz;
  const int i0 = (blockIdx.x * NW + warp) * R;
  const int k0 = (blockIdx.y * 32 + lane) * V;
  const bool col_ok = k0 < nz;
  // a strip wholly inside the grid takes the copies and results without range
  // tests (uniform over the warp)
  const bool inner = i0 > 0 && i0 + R < nr && (int)(blockIdx.y + 1) * 32 * V <= nz;
  const int off0 = (i0 - 1) * a.pitch + k0;  // row i0 - 1 (grids have fewer than 2^31 nodes)
  // the chunk's selected right-hand sides, their parity and beta
  if (warp == 0) {
    const int mm = blockIdx.z * chunk + lane;
    const bool sel = lane < chunk && mm < a.m && rhs_selected(a.st, a.mask, mm);
    const unsigned mask = __ballot_sync(0xffffffffu, sel);
    if (sel) {
      const int c = __popc(mask & ((1u << lane) - 1));
      s_m[c] = mm;
      s_odd[c] = (MODE == kStencilPcg || MODE == kStencilPcgP) ? a.st[mm].iters & 1 : 0;
      s_beta[c] = MODE == kStencilPcg ? (T)a.st[mm].beta : T(0);
    }
    if (lane == 0) s_n = __popc(mask);
  }
  __syncthreads();
  const int n = s_n;
  if (n == 0) return;
  T *ring = reinterpret_cast<T *>(ssm + warp * S::warp_bytes(chunk));
  // rows i0 - 1 .. i0 + R of the c-th right-hand side's grid function (mode Pcg:
  // z and, unless beta is 0 (p_1 = z), p_old), and nodes k0 - 1 (lane 0) and
  // k0 + V (lane 31) of rows i0 .. i0 + R - 1
  auto issue = [&](int c) {
    if (c < n) {
      T *st = ring + (c % S::stages) * S::stage;
      const size_t base = (size_t)s_m[c] * (size_t)a.field;
      const T *src[2] = {a.in, nullptr};
      if (MODE == kStencilPcg) src[1] = s_beta[c] != T(0) ? (s_odd[c] ? a.pb : a.pa) : nullptr;
      else if (MODE == kStencilPcgP) src[0] = s_odd[c] ? a.pa : a.pb;
#pragma unroll
      for (int q = 0; q < S::arrays; ++q) {
        if (src[q] == nullptr) continue;
        T *dst = st + q * S::array;
        const T *g = src[q] + base + off0;
        if (inner) {
#pragma unroll
          for (int j = 0; j < R + 2; ++j) cp_async<16>(dst + j * S::row + lane * V, g + j * a.pitch, true);
        } else {
#pragma unroll
          for (int j = 0; j < R + 2; ++j) {
            const int i = i0 - 1 + j;
            const bool ok = col_ok && i >= 0 && i < nr;
            cp_async<16>(dst + j * S::row + lane * V, ok ? g + j * a.pitch : src[q], ok);
          }
        }
        if (lane == 0 || lane == 31) {
          const int d = lane == 0 ? -1 : V, k = k0 + d;
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const bool ok = k >= 0 && k < nz && i0 + j < nr;
            cp_async<sizeof(T)>(dst + (R + 2) * S::row + 2 * j + (lane == 31),
                                ok ? g + (j + 1) * a.pitch + d : src[q], ok);
          }
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int c = 0; c < S::stages - 1; ++c) issue(c);
  T cr[R + 1][V], cz[R][V], w[R][V], czlast[R];
  auto load_coefs = [&](int mm) {
    const T *__restrict__ CR = a.CR + (size_t)mm * a.cstride;
    const T *__restrict__ CZ = a.CZ + (size_t)mm * a.czstride;
    const T *__restrict__ Wc = a.W + (size_t)mm * a.cstride;
#pragma unroll
    for (int e = 0; e < V; ++e) cr[0][e] = T(0);  // no flux through the axis
    if (col_ok && i0 > 0 && i0 <= nr) load_vec<T>(CR + (size_t)(i0 - 1) * a.pitch + k0, cr[0]);
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int i = i0 + j;
#pragma unroll
      for (int e = 0; e < V; ++e) {
        cr[j + 1][e] = T(0);
        cz[j][e] = T(0);
        w[j][e] = T(0);
      }
      czlast[j] = T(0);
      if (i >= nr) continue;
      if (col_ok) {
        load_vec<T>(CR + (size_t)i * a.pitch + k0, cr[j + 1]);
        load_vec<T>(Wc + (size_t)i * a.pitch + k0, w[j]);
      }
      // faces run to index nz, so the lane just past the last node still loads
      // its first face (the upper face of node nz - 1, fetched by the shuffle)
      if (k0 <= nz) load_vec<T>(CZ + (size_t)i * a.pitchz + k0, cz[j]);
      if (lane == 31 && k0 + V <= nz) czlast[j] = CZ[(size_t)i * a.pitchz + k0 + V];
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const T up = __shfl_down_sync(0xffffffffu, cz[j][0], 1);
      if (lane != 31) czlast[j] = up;
    }
  };
  load_coefs(s_m[0]);
  for (int c = 0; c < n; ++c) {
    T ph[R][V];  // phi, requested before the wait for this right-hand side's rows
    if (MODE == kStencilCheb) {
#pragma unroll
      for (int j = 0; j < R; ++j) {
#pragma unroll
        for (int e = 0; e < V; ++e) ph[j][e] = T(0);
        if (col_ok && i0 + j < nr)
          load_vec<T>(a.phi + (size_t)s_m[c] * (size_t)a.field + off0 + (j + 1) * a.pitch, ph[j]);
      }
    }
    asm volatile("cp.async.wait_group %0;" ::"n"(S::stages - 2) : "memory");
    __syncwarp();
    issue(c + S::stages - 1);  // into the stage read before this one
    const int m = s_m[c];
    if (c > 0 && a.cstride != 0) load_coefs(m);  // a stacked group: each its own operator
    const T *st = ring + (c % S::stages) * S::stage;
    const size_t base = (size_t)m * (size_t)a.field;
    const T beta = s_beta[c];
    const bool add_old = MODE == kStencilPcg && beta != T(0);
    T p[R + 2][V], edge[R];  // edge: node k0 - 1 in lane 0, k0 + V in lane 31
#pragma unroll
    for (int j = 0; j < R + 2; ++j) load_vec<T>(st + j * S::row + lane * V, p[j]);
#pragma unroll
    for (int j = 0; j < R; ++j) edge[j] = st[(R + 2) * S::row + 2 * j + (lane == 31)];
    if (add_old) {
      const T *so = st + S::array;
#pragma unroll
      for (int j = 0; j < R + 2; ++j) {
        T po[V];
        load_vec<T>(so + j * S::row + lane * V, po);
#pragma unroll
        for (int e = 0; e < V; ++e) p[j][e] += beta * po[e];
      }
#pragma unroll
      for (int j = 0; j < R; ++j) edge[j] += beta * so[(R + 2) * S::row + 2 * j + (lane == 31)];
    }
    // z may hold anything in its padding columns (the tensor-core path keeps
    // mode-major data in the same buffer)
    if (!inner) {
#pragma unroll
      for (int j = 0; j < R + 2; ++j)
#pragma unroll
        for (int e = 0; e < V; ++e)
          if (k0 + e >= nz) p[j][e] = T(0);
    }
    T *p_new = MODE == kStencilPcg ? (s_odd[c] ? a.pa : a.pb) : nullptr;
    T acc = T(0);  // FP32: 8 terms per thread; combined in FP64
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int i = i0 + j;
      T l = __shfl_up_sync(0xffffffffu, p[j + 1][V - 1], 1);
      T r = __shfl_down_sync(0xffffffffu, p[j + 1][0], 1);
      if (lane == 0) l = edge[j];
      if (lane == 31) r = edge[j];
      T o[V];
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const T yl = (e == 0) ? l : p[j + 1][e - 1];
        const T yr = (e == V - 1) ? r : p[j + 1][e + 1];
        const T czh = (e == V - 1) ? czlast[j] : cz[j][e + 1];
        const T y = p[j + 1][e];
        T v = w[j][e] * y;
        v = fma(cr[j + 1][e], y - p[j + 2][e], v);
        v = fma(cr[j][e], y - p[j][e], v);
        v = fma(czh, y - yr, v);
        v = fma(cz[j][e], y - yl, v);
        o[e] = v;
      }
      if (!inner) {
#pragma unroll
        for (int e = 0; e < V; ++e)
          if (k0 + e >= nz) o[e] = T(0);
        if (!col_ok || i >= nr) continue;
      }
      const size_t ro = base + off0 + (j + 1) * a.pitch;
      if (MODE == kStencilApply) {
        store_vec<T>(a.out + ro, o);
      } else if (MODE == kStencilPcg || MODE == kStencilPcgP) {
        if (MODE == kStencilPcg) store_vec<T>(p_new + ro, p[j + 1]);
        store_vec<T>(a.out + ro, o);
#pragma unroll
        for (int e = 0; e < V; ++e) acc = fma(p[j + 1][e], o[e], acc);
      } else {
        T res[V];
#pragma unroll
        for (int e = 0; e < V; ++e) {
          res[e] = (k0 + e < nz) ? o[e] - ph[j][e] : T(0);
          acc = fma(res[e], res[e], acc);
        }
        store_vec<T>(a.out + ro, res);
      }
    }
    if (MODE != kStencilApply) s_acc[c][threadIdx.x] = acc;
  }
  if (MODE == kStencilApply) return;
  // a warp per right-hand side: its partial (the threads' sums, a fixed order)
  // and the CTA's arrival for it; then the scalar steps of those this CTA is
  // last of
  const unsigned nb = gridDim.x * gridDim.y;
  __syncthreads();
  for (int c = warp; c < n; c += NW) {
    T v[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) v[i] = s_acc[c][i * 32 + lane];
    const double tot = warp_sum_fp32(v);
    if (lane == 0) {
      if (a.partial != nullptr)
        a.partial[(size_t)s_m[c] * kPartialStride + blockIdx.y * gridDim.x + blockIdx.x] = tot;
      s_last[c] = a.fin.kind != kFinNone && finish_arrive(a.fin, s_m[c], nb);
    }
  }
  if (a.fin.kind == kFinNone) return;
  __syncthreads();
  for (int c = 0; c < n; ++c)
    if (s_last[c])
      finish_last(a.fin, s_m[c], a.partial ? a.partial + (size_t)s_m[c] * kPartialStride : nullptr, (int)nb, red);
}

// 16 rows per CTA, walked down with a three-row register window: every element
// is read once plus one halo row per CTA edge.  For grids on which the strips'
// partials would not fit their array (see strip_warps).
template <typename T, int MODE>
__global__ void __launch_bounds__(256) stencil_kernel(const StencilArgs<T> a, int rows) {
  constexpr int V = VecT<T>::n;
  __shared__ double red[8];
  const int m = blockIdx.x;
  if (!rhs_selected(a.st, a.mask, m)) return;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  const int k0 = ((blockIdx.z * nwarps + warp) * 32 + lane) * V;
  const int nr = a.nr, nz = a.nz;
  const int i0 = blockIdx.y * rows;
  const int i1 = min(i0 + rows, nr);
  const size_t base = (size_t)m * (size_t)a.field;
  const bool col_ok = k0 < nz;
  const T *__restrict__ CR = a.CR + (size_t)m * a.cstride;
  const T *__restrict__ CZ = a.CZ + (size_t)m * a.czstride;
  const T *__restrict__ Wc = a.W + (size_t)m * a.cstride;
  T beta = T(0);
  const T *p_old = nullptr;
  T *p_new = nullptr;
  const T *src = a.in;  // the grid function (before the direction update in mode Pcg)
  if (MODE == kStencilPcg) {
    beta = (T)a.st[m].beta;
    const bool odd = a.st[m].iters & 1;
    p_old = odd ? a.pb : a.pa;
    p_new = odd ? a.pa : a.pb;
  } else if (MODE == kStencilPcgP) {
    src = (a.st[m].iters & 1) ? a.pa : a.pb;
  }

  auto load_row = [&](int i, T (&v)[V]) {
#pragma unroll
    for (int e = 0; e < V; ++e) v[e] = T(0);
    if (!col_ok) return;
    const size_t off = base + (size_t)i * a.pitch + k0;
    T t[V];
    load_vec<T>(src + off, t);
    if (MODE == kStencilPcg && beta != T(0)) {
      T po[V];
      load_vec<T>(p_old + off, po);
#pragma unroll
      for (int e = 0; e < V; ++e) t[e] += beta * po[e];
    }
#pragma unroll
    for (int e = 0; e < V; ++e) v[e] = (k0 + e < nz) ? t[e] : T(0);
  };
  auto load_coef = [&](const T *c, int i, T (&v)[V]) {
#pragma unroll
    for (int e = 0; e < V; ++e) v[e] = T(0);
    if (!col_ok) return;
    load_vec<T>(c + (size_t)i * a.pitch + k0, v);
  };

  // Everything row i + 1 needs (values, its CR / CZ / W rows and the two
  // warp-edge halo values) is loaded one row ahead, while row i is computed.
  auto load_halo = [&](int i, T &left, T &right, T &czlast) {
    const size_t rowoff = base + (size_t)i * a.pitch;
    left = right = czlast = T(0);
    if (lane == 0 && col_ok && k0 > 0) left = StencilValue<T, MODE>::at(src, p_old, rowoff + k0 - 1, beta);
    if (lane == 31) {
      if (k0 + V < nz) right = StencilValue<T, MODE>::at(src, p_old, rowoff + k0 + V, beta);
      if (k0 + V <= nz) czlast = CZ[(size_t)i * a.pitchz + k0 + V];
    }
  };
  auto load_cz = [&](int i, T (&v)[V]) {
#pragma unroll
    for (int e = 0; e < V; ++e) v[e] = T(0);
    // Faces run to index nz, so the lane just past the last node still loads
    // its first face (the upper face of node nz - 1, fetched by the shuffle).
    if (k0 <= nz) load_vec<T>(CZ + (size_t)i * a.pitchz + k0, v);
  };

  // every row of the DRAM stream(s) this CTA reads, into L2 at once: the
  // register loads below then wait on L2 instead of DRAM
  if (col_ok)
    for (int i = max(i0 - 1, 0); i <= i1 && i < nr; ++i) {
      const size_t off = base + (size_t)i * a.pitch + k0;
      prefetch_l2(src + off);
      if (MODE == kStencilPcg) prefetch_l2(p_old + off);
      if ((MODE == kStencilResidual || MODE == kStencilCheb) && i >= i0 && i < i1) prefetch_l2(a.phi + off);
    }
  T pm[V], pc[V], pn[V], crl[V], crh[V], czl[V], w[V];
  T left, right, czlast;
  if (i0 > 0) {
    load_row(i0 - 1, pm);
    load_coef(CR, i0 - 1, crl);
  } else {
#pragma unroll
    for (int e = 0; e < V; ++e) { pm[e] = T(0); crl[e] = T(0); }
  }
  load_row(i0, pc);
  load_coef(CR, i0, crh);
  load_cz(i0, czl);
  load_coef(Wc, i0, w);
  load_halo(i0, left, right, czlast);

  // FP32 partials per thread are short sums (<= 64 terms); the CTA and grid
  // combination is FP64.
  T acc = T(0);
  for (int i = i0; i < i1; ++i) {
    T crn[V], czn[V], wn[V], leftn = T(0), rightn = T(0), czlastn = T(0);
    if (i + 1 < nr) {
      load_row(i + 1, pn);
    } else {
#pragma unroll
      for (int e = 0; e < V; ++e) pn[e] = T(0);
    }
    if (i + 1 < i1) {
      load_coef(CR, i + 1, crn);
      load_cz(i + 1, czn);
      load_coef(Wc, i + 1, wn);
      load_halo(i + 1, leftn, rightn, czlastn);
    } else {
#pragma unroll
      for (int e = 0; e < V; ++e) crn[e] = czn[e] = wn[e] = T(0);
    }
    const size_t rowoff = base + (size_t)i * a.pitch;
    // z-neighbours of the lane's first and last node.
    T l = __shfl_up_sync(0xffffffffu, pc[V - 1], 1);
    T r = __shfl_down_sync(0xffffffffu, pc[0], 1);
    T czh_last = __shfl_down_sync(0xffffffffu, czl[0], 1);
    if (lane == 0) l = left;
    if (lane == 31) {
      r = right;
      czh_last = czlast;
    }

    T o[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const T yl = (e == 0) ? l : pc[e - 1];
      const T yr = (e == V - 1) ? r : pc[e + 1];
      const T czh = (e == V - 1) ? czh_last : czl[e + 1];
      const T y = pc[e];
      T v = w[e] * y;
      v = fma(crh[e], y - pn[e], v);
      v = fma(crl[e], y - pm[e], v);
      v = fma(czh, y - yr, v);
      v = fma(czl[e], y - yl, v);
      o[e] = (k0 + e < nz) ? v : T(0);
    }
    if (col_ok) {
      if (MODE == kStencilApply) {
        store_vec<T>(a.out + rowoff + k0, o);
      } else if (MODE == kStencilPcg || MODE == kStencilPcgP) {
        if (MODE == kStencilPcg) store_vec<T>(p_new + rowoff + k0, pc);
        store_vec<T>(a.out + rowoff + k0, o);
#pragma unroll
        for (int e = 0; e < V; ++e) acc = fma(pc[e], o[e], acc);
      } else {
        T ph[V];
        load_vec<T>(a.phi + rowoff + k0, ph);
        T res[V];
#pragma unroll
        for (int e = 0; e < V; ++e) {
          res[e] = (k0 + e < nz) ? ((MODE == kStencilResidual) ? ph[e] - o[e] : o[e] - ph[e]) : T(0);
          acc = fma(res[e], res[e], acc);
        }
        if (MODE == kStencilResidual) {
          if (a.out_res) store_vec<T>(a.out_res + rowoff + k0, res);
          if (a.out32) {
            *reinterpret_cast<float2 *>(a.out32 + rowoff + k0) = make_float2((float)res[0], (float)res[1]);
          }
        } else {
          store_vec<T>(a.out + rowoff + k0, res);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < V; ++e) {
      pm[e] = pc[e];
      pc[e] = pn[e];
      crl[e] = crh[e];
      crh[e] = crn[e];
      czl[e] = czn[e];
      w[e] = wn[e];
    }
    left = leftn;
    right = rightn;
    czlast = czlastn;
  }
  if (MODE != kStencilApply) {
    if (a.partial != nullptr) {  // uniform over the CTA
      const double s = block_sum_of(acc, red);
      if (threadIdx.x == 0)
        a.partial[(size_t)m * kPartialStride + blockIdx.y * gridDim.z + blockIdx.z] = s;
    } else {
      __syncthreads();  // every warp has read the state before this CTA arrives
    }
    const int nb = (int)(gridDim.y * gridDim.z);
    finish_rhs(a.fin, m, (unsigned)nb, a.partial ? a.partial + (size_t)m * kPartialStride : nullptr, nb, red);
  }
}

// ---- double-float residual -------------------------------------------------
// Pairs (h, l) of FP32 numbers carry about 48 significant bits: sums by Knuth's
// two-sum, products by the FMA two-product (the exact error of a*b is
// fma(a, b, -a*b)).  GB300 runs FP32 about 58 times faster than FP64, so the
// true residual of the mixed method costs a few FP32 operations per flop
// instead of FP64 ones.
struct DF {
  float h, l;
};
__device__ __forceinline__ DF df_two_sum(float a, float b) {
  const float s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}

// One pass does what were two (x += x32 in double-float, then the residual of
// the new x): each warp advances x on its own 2 rows and forms the advanced x of
// the rows and columns around them again from the old pair, so no CTA waits for
// another.  All loads of a strip are issued before the first use; about 120
// FP32 operations per node follow.  NW warps per CTA (see df_warps), 128
// registers a thread.
template <bool FOLD, int NW>
__global__ void __launch_bounds__(32 * NW, 16 / NW) residual_df_kernel(const DfResidualArgs a) {
  __shared__ double red[NW];
  const int nr = a.nr, nz = a.nz, P = a.pitch, PZ = a.pitchz, lane = threadIdx.x & 31;
  const int k0 = (blockIdx.y * 32 + lane) * 4;
  const int i0 = (blockIdx.x * NW + (threadIdx.x >> 5)) * 2;
  const bool col_ok = k0 < nz;
  // right-hand sides blockIdx.z, + gridDim.z, ... (at most 32), those selected:
  // one CTA per right-hand side would launch 16 times as many CTAs as do work
  // in an iteration in which few are due
  const int mine = blockIdx.z + lane * gridDim.z;
  unsigned todo = __ballot_sync(0xffffffffu, mine < a.m && rhs_selected(a.st, a.mask, mine));
  for (; todo != 0; todo &= todo - 1) {
  const int m = blockIdx.z + (__ffs(todo) - 1) * gridDim.z;
  const size_t base = (size_t)m * (size_t)a.field;
  const int nrep = FOLD ? (int)a.st[m].tmp : 0, sel = nrep & 1;
  const bool have_x = !(FOLD && a.zero_start && nrep == 0);
  const float *xh = a.xh[sel] + base, *xl = a.xl[sel] + base, *xd = FOLD ? a.d + base : nullptr;
  float *nh = a.xh[sel ^ 1] + base, *nl = a.xl[sel ^ 1] + base;
  const float *crh = a.CRh + (size_t)m * a.cstride, *crl = a.CRl + (size_t)m * a.cstride;
  const float *czh = a.CZh + (size_t)m * a.czstride, *czl = a.CZl + (size_t)m * a.czstride;
  const float *wh = a.Wh + (size_t)m * a.cstride, *wl = a.Wl + (size_t)m * a.cstride;
  // x + d as a pair (two-sum, then renormalised)
  auto fold = [](float x, float lo, float c, float &h, float &l) {
    const float s = x + c, bb = s - x;
    const float err = ((x - (s - bb)) + (c - bb)) + lo;
    h = s + err;
    l = err - (h - s);
  };
  // 4 consecutive values of a row (zero outside the grid; padding columns hold
  // zeros)
  auto ld4 = [&](const float *p, size_t off, bool ok, float (&v)[4]) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    if (ok) t = *reinterpret_cast<const float4 *>(p + off);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  };
  // x of rows i0 - 1 .. i0 + 2, and the strip's neighbours of rows i0, i0 + 1
  // (lane 0: node k0 - 1; lane 31: node k0 + 4)
  float yh[4][4], yl[4][4], d[4][4], eh[2], el[2], ed[2];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int i = i0 - 1 + j;
    const bool ok = col_ok && i >= 0 && i < nr;
    const size_t off = (size_t)i * P + k0;
    ld4(xh, off, ok && have_x, yh[j]);
    ld4(xl, off, ok && have_x, yl[j]);
    if (FOLD) ld4(xd, off, ok, d[j]);
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int ke = lane == 0 ? k0 - 1 : k0 + 4;
    const bool eok = i0 + j < nr && (lane == 0 || lane == 31) && ke >= 0 && ke < nz;
    const size_t eo = (size_t)(i0 + j) * P + ke;
    eh[j] = eok && have_x ? xh[eo] : 0.f;
    el[j] = eok && have_x ? xl[eo] : 0.f;
    ed[j] = FOLD && eok ? xd[eo] : 0.f;
  }
  if (FOLD) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) fold(yh[j][e], yl[j][e], d[j][e], yh[j][e], yl[j][e]);
#pragma unroll
    for (int j = 0; j < 2; ++j) fold(eh[j], el[j], ed[j], eh[j], el[j]);
  }
  float cph[4], cpl[4];  // CR_{i-1}: 0 on the axis
  ld4(crh, (size_t)(i0 - 1) * P + k0, col_ok && i0 > 0 && i0 <= nr, cph);
  ld4(crl, (size_t)(i0 - 1) * P + k0, col_ok && i0 > 0 && i0 <= nr, cpl);
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int i = i0 + j;
    const bool ok = col_ok && i < nr;
    const size_t ro = (size_t)i * P + k0, zo = (size_t)i * PZ + k0;
    float ch[4], cl[4], w4h[4], w4l[4], zh[4], zl[4], fh[4], fl[4];
    ld4(crh, ro, ok, ch);
    ld4(crl, ro, ok, cl);
    ld4(wh, ro, ok, w4h);
    ld4(wl, ro, ok, w4l);
    ld4(czh, zo, ok, zh);  // faces k0 .. k0 + 3
    ld4(czl, zo, ok, zl);
    ld4(a.ph + base, ro, ok, fh);
    ld4(a.pl + base, ro, ok, fl);
    const bool up = ok && k0 + 4 <= nz;  // face k0 + 4
    const DF z4 = {up ? czh[zo + 4] : 0.f, up ? czl[zo + 4] : 0.f};
    // z-neighbours outside the 4 nodes
    DF yleft = {__shfl_up_sync(0xffffffffu, yh[j + 1][3], 1), __shfl_up_sync(0xffffffffu, yl[j + 1][3], 1)};
    DF yright = {__shfl_down_sync(0xffffffffu, yh[j + 1][0], 1), __shfl_down_sync(0xffffffffu, yl[j + 1][0], 1)};
    if (lane == 0) yleft = {eh[j], el[j]};
    if (lane == 31) yright = {eh[j], el[j]};
    float res[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const DF y = {yh[j + 1][e], yl[j + 1][e]};
      const DF ylf = (e == 0) ? yleft : DF{yh[j + 1][e - 1], yl[j + 1][e - 1]};
      const DF yr = (e == 3) ? yright : DF{yh[j + 1][e + 1], yl[j + 1][e + 1]};
      const DF czlo = {zh[e], zl[e]};
      const DF czhi = (e == 3) ? z4 : DF{zh[e + 1], zl[e + 1]};
      // r = phi - A y, A y = W y + CR_i (y - y_{i+1}) + CR_{i-1} (y - y_{i-1})
      //                     + CZ_{k+1} (y - y_{k+1}) + CZ_k (y - y_{k-1}),
      // as a compensated sum (Ogita, Rump and Oishi's Dot2: each product's
      // high part exact by the FMA two-product, each addition's error by
      // two-sum, the small terms gathered in one FP32 word): the accuracy of
      // double-float arithmetic without renormalising after every operation
      float sh = fh[e], se = fl[e];
      auto sub_prod = [&](float ph, float pl, float dh, float dl) {  // s -= (ph + pl)(dh + dl)
        const float p = ph * dh;
        const float pe = fmaf(ph, dh, -p);
        const float lo = fmaf(ph, dl, fmaf(pl, dh, pe));
        const float t = sh - p, bb = t - sh;
        se += ((sh - (t - bb)) - (p + bb)) - lo;
        sh = t;
      };
      // y - y_n as an unnormalised pair: the high parts by two-sum, the low
      // parts' difference added to its error
      auto diff = [](DF u, DF w, float &dh, float &dl) {
        const DF s2 = df_two_sum(u.h, -w.h);
        dh = s2.h;
        dl = s2.l + (u.l - w.l);
      };
      float dh, dl;
      sub_prod(w4h[e], w4l[e], y.h, y.l);
      diff(y, DF{yh[j + 2][e], yl[j + 2][e]}, dh, dl);
      sub_prod(ch[e], cl[e], dh, dl);
      diff(y, DF{yh[j][e], yl[j][e]}, dh, dl);
      sub_prod(cph[e], cpl[e], dh, dl);
      diff(y, yr, dh, dl);
      sub_prod(czhi.h, czhi.l, dh, dl);
      diff(y, ylf, dh, dl);
      sub_prod(czlo.h, czlo.l, dh, dl);
      res[e] = (ok && k0 + e < nz) ? sh + se : 0.f;
      acc = fmaf(res[e], res[e], acc);
    }
    if (ok) {
      *reinterpret_cast<float4 *>(a.r32 + base + ro) = make_float4(res[0], res[1], res[2], res[3]);
      if (FOLD) {
        *reinterpret_cast<float4 *>(nh + ro) = make_float4(yh[j + 1][0], yh[j + 1][1], yh[j + 1][2], yh[j + 1][3]);
        *reinterpret_cast<float4 *>(nl + ro) = make_float4(yl[j + 1][0], yl[j + 1][1], yl[j + 1][2], yl[j + 1][3]);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      cph[e] = ch[e];
      cpl[e] = cl[e];
    }
  }
  const double sum = block_sum_of(acc, red);
  const int nb = (int)(gridDim.x * gridDim.y), slot = blockIdx.y * gridDim.x + blockIdx.x;
  if (threadIdx.x == 0) a.partial[(size_t)m * kPartialStride + slot] = sum;
  finish_rhs(a.fin, m, (unsigned)nb, a.partial + (size_t)m * kPartialStride, nb, red);
  }
}

int column_warps(int nz, int vec) {
  int w = (nz + 32 * vec - 1) / (32 * vec);
  return w < kStencilWarps ? (w < 1 ? 1 : w) : kStencilWarps;
}

}  // namespace

// Warps per CTA of the strip kernel, by the grid alone (see there); 0 where its
// partials, one per CTA, would not fit the array: the 16-row kernel runs.
// FP64 (vec = 2) runs the 16-row kernel always: it is bound by the FP64 pipe, and
// strips form p = z + beta p_old twice on their shared rows (500 x 511 x 8: 81 us
// against 64).
static int strip_warps(int nr, int nz, int vec, int *gx, int *gy) {
  if (vec != 4) return 0;
  *gy = (nz + 32 * vec - 1) / (32 * vec);
  const int strips = (nr + kStripRows - 1) / kStripRows;
  const long long all = (long long)strips * *gy;
  const int nw = all >= 2048 ? 8 : all >= 512 ? 4 : 2;
  *gx = (strips + nw - 1) / nw;
  return (long long)*gx * *gy <= kPartialStride ? nw : 0;
}

// Rows per CTA of stencil_kernel, by the grid alone (its partials' order): 16, or
// down to 4 while one right-hand side fills less than two CTAs per SM: a CTA walks
// its rows one memory round trip after the other, and more of them hide it.  FP64
// PCG pass, cold caches, 16 rows and 4: 500 x 511, one right-hand side 43 and 18 us,
// eight 72 and 68 (there the FP64 pipe bounds it).
static int long_rows(int nr, int nz, int vec) {
  const int wx = column_warps(nz, vec), gz = (nz + 32 * vec * wx - 1) / (32 * vec * wx);
  int rows = kRowsLong;
  while (rows > 4 && (long long)((nr + rows - 1) / rows) * gz < 304) rows /= 2;
  return rows;
}

int stencil_blocks_per_rhs(int nr, int nz, int vec) {
  int sx, sy;
  if (strip_warps(nr, nz, vec, &sx, &sy)) return sx * sy;
  const int wx = column_warps(nz, vec), rows = long_rows(nr, nz, vec);
  const int gz = (nz + 32 * vec * wx - 1) / (32 * vec * wx);
  return (nr + rows - 1) / rows * gz;
}

template <typename T, int MODE>
static void launch_stencil_mode(const StencilArgs<T> &a, cudaStream_t s) {
  constexpr int V = VecT<T>::n;
  int sx, sy;
  const int nw = strip_warps(a.nr, a.nz, V, &sx, &sy);
  note_launch();
  if constexpr (V == 4) if (nw != 0) {
    // right-hand sides per CTA: as many as leave two rounds of 24 resident warps
    // on each of 152 SMs
    const long long c = (long long)a.m * sx * sy * nw / (152 * 48);
    const int chunk = a.cstride != 0 ? 1 : (int)std::max<long long>(1, std::min<long long>(c, kStripChunk));
    const dim3 grid(sx, sy, (a.m + chunk - 1) / chunk);
    const size_t smem = nw * StripShape<T, MODE>::warp_bytes(chunk);
    if (nw == 8) {
      ensure_smem_attr((const void *)strip_kernel<T, MODE, 8>, smem);
      strip_kernel<T, MODE, 8><<<grid, 256, smem, s>>>(a, chunk);
    } else if (nw == 4) {
      ensure_smem_attr((const void *)strip_kernel<T, MODE, 4>, smem);
      strip_kernel<T, MODE, 4><<<grid, 128, smem, s>>>(a, chunk);
    } else {
      strip_kernel<T, MODE, 2><<<grid, 64, smem, s>>>(a, chunk);
    }
    return;
  }
  const int wx = column_warps(a.nz, V), rows = long_rows(a.nr, a.nz, V);
  const dim3 grid(a.m, (a.nr + rows - 1) / rows, (a.nz + 32 * V * wx - 1) / (32 * V * wx));
  stencil_kernel<T, MODE><<<grid, 32 * wx, 0, s>>>(a, rows);
}

template <typename T>
void launch_stencil(int mode, const StencilArgs<T> &a, cudaStream_t s) {
  switch (mode) {
    case kStencilApply: launch_stencil_mode<T, kStencilApply>(a, s); break;
    case kStencilPcg: launch_stencil_mode<T, kStencilPcg>(a, s); break;
    case kStencilPcgP: launch_stencil_mode<T, kStencilPcgP>(a, s); break;
    case kStencilResidual:  // FP64 only (the mixed PCG's is launch_residual_df)
      if constexpr (sizeof(T) == 8) launch_stencil_mode<T, kStencilResidual>(a, s);
      break;
    default: launch_stencil_mode<T, kStencilCheb>(a, s); break;
  }
}

// Warps per residual CTA, by the grid alone: 4 (few right-hand sides are due at
// a time: small CTAs spread them) while that gives at most 2048 partials for the
// last CTA to sum, more on larger grids.
static int df_warps(int nr, int nz, int *gx, int *gy) {
  *gy = (nz + 127) / 128;
  int nw = 4;
  for (;; nw *= 2) {
    *gx = ((nr + 1) / 2 + nw - 1) / nw;
    if (nw == 16 || *gx * *gy <= (nw == 4 ? 2048 : 8192)) return nw;
  }
}

int residual_df_blocks(int nr, int nz) {
  int gx, gy;
  df_warps(nr, nz, &gx, &gy);
  return gx * gy;
}

template <bool FOLD>
static void launch_df(const DfResidualArgs &a, cudaStream_t s) {
  int gx, gy;
  const int nw = df_warps(a.nr, a.nz, &gx, &gy);
  const dim3 grid(gx, gy, std::max(std::min(a.m, 4), (a.m + 31) / 32));
  note_launch();
  if (nw == 4) residual_df_kernel<FOLD, 4><<<grid, 128, 0, s>>>(a);
  else if (nw == 8) residual_df_kernel<FOLD, 8><<<grid, 256, 0, s>>>(a);
  else residual_df_kernel<FOLD, 16><<<grid, 512, 0, s>>>(a);
}

void launch_residual_df(const DfResidualArgs &a, cudaStream_t s) {
  if (a.d != nullptr) launch_df<true>(a, s);
  else launch_df<false>(a, s);
}

template void launch_stencil<float>(int, const StencilArgs<float> &, cudaStream_t);
template void launch_stencil<double>(int, const StencilArgs<double> &, cudaStream_t);

}  // namespace ax
