// Segmented reductions and updates of flexible GMRES(m) (paper Sec. 3.2,
// GMRES) on sm_103a; fs_orth.cu holds the orthogonalisation.
//
// A problem holds one or more independent instances ("segments": the
// instances of a batch, or the single mesh of an ordinary problem).  Every
// segment runs its own Arnoldi process: its own Hessenberg matrix, Givens
// rotations, convergence flag and update, so a segment's iterates do not
// depend on the other segments.  Vectors are walked through a work-list of
// tiles, each a contiguous range of one segment (at most kTileLen entries);
// one thread block per tile.  Per-tile partial sums go to scratch; the last
// tile of a segment to finish (per-segment atomic ticket, never waited on)
// reduces them in FP64.  Kernels that span all segments (SpMV, multigrid)
// skip their work once every segment has converged (KCtl::all_done).
#include <cuda_runtime.h>

#include <cmath>

#include <type_traits>

#include "fs_device.h"

namespace fs {

namespace {

constexpr unsigned kFull = 0xffffffffu;
// threads per tile block: few blocks (one per tile), so each brings many warps
constexpr int kKB = 512;

template <typename V>
__device__ __forceinline__ V warp_sum(V v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
  return v;
}

// Block sum (all threads participate); valid in every thread afterwards.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sm[kKB / 32];
  __shared__ double total;
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sm[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int i = 0; i < kKB / 32; ++i) t += sm[i];
    total = t;
  }
  __syncthreads();
  return total;
}

// True in every thread of the last tile block of its segment to arrive.
__device__ __forceinline__ bool last_of_segment(unsigned* counter, int ntiles) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == (unsigned)(ntiles - 1);
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Sum of partial[v * ntiles_total + t] over the segment's tiles, for v <
// nvec; result in res[v] (shared), all threads of the block participate.
// A warp per vector; a lane reads its tiles four at a time (loads from L2,
// where the other blocks' partials are visible after the ticket) into four
// sums, added in a fixed order.
__device__ void reduce_segment(const double* partial, int64_t stride, int first, int count,
                               int nvec, double* res) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int v = w; v < nvec; v += nw) {
    const double* p = partial + (int64_t)v * stride + first;
    double s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    int t = lane;
    for (; t + 96 < count; t += 128) {
      const double a0 = __ldcg(p + t), a1 = __ldcg(p + t + 32), a2 = __ldcg(p + t + 64),
                   a3 = __ldcg(p + t + 96);
      s0 += a0;
      s1 += a1;
      s2 += a2;
      s3 += a3;
    }
    for (; t < count; t += 32) s0 += __ldcg(p + t);
    double s = warp_sum((s0 + s1) + (s2 + s3));
    if (lane == 0) res[v] = s;
  }
  __syncthreads();
}

// field: 0 beta, 1 bnorm, 2 rnorm
template <typename V>
__global__ void __launch_bounds__(kKB) k_seg_norm(const V* __restrict__ x, const Tile* tiles,
                                                  int ntiles, SegState* st, double* partial,
                                                  int field) {
  pdl_wait();
  const Tile t = tiles[blockIdx.x];
  SegState& S = st[t.seg];
  double acc = 0;
  for (int e = threadIdx.x; e < t.len; e += kKB) {
    const double v = (double)x[t.start + e];
    acc += v * v;
  }
  const double bs = block_sum(acc);
  if (threadIdx.x == 0) partial[blockIdx.x] = bs;
  if (!last_of_segment(&S.counter[4 + field], S.ntiles)) return;
  __shared__ double res[1];
  reduce_segment(partial, ntiles, S.first_tile, S.ntiles, 1, res);
  if (threadIdx.x == 0) {
    const double n = sqrt(res[0]);
    if (field == 0) S.beta = n;
    else if (field == 1) S.bnorm = n;
    else S.rnorm = n;
    S.counter[4 + field] = 0;
  }
}

// Start of a restart cycle: tolerances, right-hand side of the least-squares
// problem, done flags (converged, retired by the host, or non-finite).
// tol_abs = rtol * (relative_to_beta ? beta : bnorm).
__global__ void k_seg_cycle_init(SegState* st, KCtl* ctl, int relative_to_beta,
                                 cudaGraphConditionalHandle cond) {
  pdl_wait();
  __shared__ int ndone;
  if (threadIdx.x == 0) ndone = 0;
  __syncthreads();
  const int m = ctl->m;
  for (int s = threadIdx.x; s < ctl->nseg; s += blockDim.x) {
    SegState& S = st[s];
    const double beta = S.beta;
    S.tol_abs = S.rtol * (relative_to_beta ? beta : S.bnorm);
    S.k = 0;
    S.bad = isfinite(beta) ? 0 : 1;
    S.resid = beta;
    for (int i = 0; i <= m; ++i) S.g[i] = 0.0;
    S.g[0] = beta;
    S.done = (S.retired || S.bad || beta <= S.tol_abs || beta == 0.0) ? 1 : 0;
    if (S.done) atomicAdd(&ndone, 1);
    for (int c = 0; c < 4; ++c) S.counter[c] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    ctl->ndone = ndone;
    ctl->all_done = ndone == ctl->nseg ? 1 : 0;
    ctl->j = 0;
    ctl->nfin = ctl->nredo = 0;
    ctl->bar = ctl->bar_base = 0;
    if (cond) cudaGraphSetConditional(cond, ndone == ctl->nseg ? 0u : 1u);
  }
}

// x *= 1 / beta of the tile's segment (skipped once done)
template <typename V>
__global__ void __launch_bounds__(kKB) k_seg_scale(JVec<V> xv, const Tile* tiles,
                                                   const SegState* st) {
  pdl_wait();
  const Tile t = tiles[blockIdx.x];
  const SegState& S = st[t.seg];
  if (S.done) return;
  V* __restrict__ x = xv.get();
  const V f = (V)(1.0 / S.beta);
  for (int e = threadIdx.x; e < t.len; e += kKB) x[t.start + e] *= f;
}

// z 2^-896 in FP64, from the bits of a finite z: an exponent field 896 lower is
// the same field, so the mantissa only moves (zeros and FP32 denormals
// included; both scales cancel exactly in a product with y 2^896).  Three
// integer operations where the conversion instruction takes as long as an
// FP64 FMA, 64 cycles of a quarter SM per warp.
__device__ __forceinline__ double widen(float z) {
  const unsigned b = __float_as_uint(z);
  return __hiloint2double((int)((b & 0x80000000u) | ((b & 0x7fffffffu) >> 3)), (int)(b << 29));
}
// The sum over the directions by conversion.  For FP32 directions that are not
// all finite it is a call: inlined, the compiler would convert beside every
// widened entry and select.
template <typename V>
__device__ __forceinline__ double sum_directions_impl(const V* __restrict__ z, int64_t n, int k,
                                                      const double* y) {
  double s[4] = {0, 0, 0, 0};
  int c = 0;
  for (; c + 4 <= k; c += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) s[u] += y[c + u] * (double)z[(int64_t)(c + u) * n];
  }
  for (; c < k; ++c) s[0] += y[c] * (double)z[(int64_t)c * n];
  return (s[0] + s[1]) + (s[2] + s[3]);
}
__device__ __forceinline__ double sum_directions(const double* z, int64_t n, int k,
                                                 const double* y) {
  return sum_directions_impl(z, n, k, y);
}
__device__ __noinline__ double sum_directions(const float* z, int64_t n, int k, const double* y) {
  return sum_directions_impl(z, n, k, y);
}

// y = H(0:k,0:k)^-1 g(0:k) of the tile's segment, then x += Z y.
//
// The back substitution runs in one warp, a lane per unknown with the
// reciprocals of the diagonal taken beforehand, from the triangle in shared
// memory (one thread walking it through global memory took most of the
// kernel's time on small vectors).  The sums over the directions run in FP64,
// FP32 directions widened by their bits (unless one is not finite, or a
// coefficient is 2^127 or more): FP64 arithmetic is what bounds the kernel (109
// us of FMAs on the 48^3 cube).  Per cycle on GB300, 24 directions or so: 78 ->
// 32 us on the 512x96 channel, 418 -> 189 on the 48^3 cube, 209 -> 107 on the
// batch of 96 squares, 48 -> 24 on the FP64 8^2 square (sums of FP32 pairs, 48
// bits, took 35, 163 and 81 us).
template <typename V, typename X>
__global__ void __launch_bounds__(kKB) k_seg_update_x(const SegState* st, const KCtl* ctl,
                                                      const V* __restrict__ Z, int64_t n,
                                                      const Tile* tiles, X* __restrict__ x) {
  pdl_wait();
  constexpr bool f32 = sizeof(V) == 4;
  __shared__ double y[kMaxRestart], ys[kMaxRestart];  // y, y 2^896
  __shared__ int by_bits;
  constexpr int kLd = 33;  // odd: a lane's row starts on a bank of its own
  __shared__ double H[kMaxRestart * kLd];
  const Tile t = tiles[blockIdx.x];
  const SegState& S = st[t.seg];
  const int k = S.k, m = ctl->m;
  if (k == 0) return;
  for (int i = threadIdx.x >> 5; i < k; i += kKB / 32) {
    const int c = threadIdx.x & 31;
    if (c < k) H[i * kLd + c] = S.H[i * m + c];
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int i = threadIdx.x;
    double g = i < k ? S.g[i] : 0.0, mine = 0.0;
    const double r = i < k ? 1.0 / H[i * kLd + i] : 0.0;
    for (int c = k - 1; c >= 0; --c) {
      const double yc = __shfl_sync(kFull, g * r, c);
      if (i < c) g -= H[i * kLd + c] * yc;
      if (i == c) mine = yc;
    }
    if (i < k) {
      y[i] = mine;
      ys[i] = scalbn(mine, 896);
    }
    const bool fit = __all_sync(kFull, fabs(mine) < 0x1p127);
    if (i == 0) by_bits = fit;
  }
  __syncthreads();
  const bool bits = f32 && by_bits;
  for (int e = threadIdx.x; e < t.len; e += kKB) {
    const int64_t i = t.start + e;
    double sum = 0.0;
    bool done = false;
    if constexpr (f32) {
      if (bits) {
        // four directions at a time into separate sums (independent loads)
        double s[4] = {0, 0, 0, 0};
        unsigned top = 0;  // largest exponent field
        int c = 0;
        for (; c + 4 <= k; c += 4) {
          float z[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) z[u] = Z[(int64_t)(c + u) * n + i];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            top = max(top, __float_as_uint(z[u]) & 0x7f800000u);
            s[u] += ys[c + u] * widen(z[u]);
          }
        }
        for (; c < k; ++c) {
          const float z = Z[(int64_t)c * n + i];
          top = max(top, __float_as_uint(z) & 0x7f800000u);
          s[0] += ys[c] * widen(z);
        }
        sum = (s[0] + s[1]) + (s[2] + s[3]);
        done = top != 0x7f800000u;  // all finite
      }
    }
    if (!done) sum = sum_directions(Z + i, n, k, y);
    x[i] = (X)((double)x[i] + sum);
  }
}

// out = in / rnorm of the segment (0 for retired segments)
template <typename A, typename B>
__global__ void __launch_bounds__(kKB) k_seg_normalise(const A* __restrict__ in,
                                                       B* __restrict__ out, const Tile* tiles,
                                                       const SegState* st) {
  pdl_wait();
  const Tile t = tiles[blockIdx.x];
  const SegState& S = st[t.seg];
  const double f = (S.retired || S.rnorm == 0.0) ? 0.0 : 1.0 / S.rnorm;
  for (int e = threadIdx.x; e < t.len; e += kKB)
    out[t.start + e] = (B)((double)in[t.start + e] * f);
}

// x += rnorm d for the segments that are still refined
template <typename V, typename X>
__global__ void __launch_bounds__(kKB) k_seg_axpy(X* __restrict__ x, const V* __restrict__ d,
                                                  const Tile* tiles, const SegState* st) {
  pdl_wait();
  const Tile t = tiles[blockIdx.x];
  const SegState& S = st[t.seg];
  if (S.retired) return;
  const double a = S.rnorm;
  for (int e = threadIdx.x; e < t.len; e += kKB)
    x[t.start + e] = (X)((double)x[t.start + e] + a * (double)d[t.start + e]);
}

}  // namespace

// ---------------------------------------------------------------------------
template <typename V>
void launch_seg_norm(const V* x, const TileList& tl, SegState* st, double* partial, int field,
                     cudaStream_t s) {
  launch_k(k_seg_norm<V>, tl.ntiles, kKB, 0, s, x, tl.tiles, tl.ntiles, st, partial, field);
  count_launches(1);
}
template void launch_seg_norm<double>(const double*, const TileList&, SegState*, double*, int,
                                      cudaStream_t);
template void launch_seg_norm<float>(const float*, const TileList&, SegState*, double*, int,
                                     cudaStream_t);

void launch_seg_cycle_init(SegState* st, KCtl* ctl, int relative_to_beta,
                           cudaGraphConditionalHandle cond, cudaStream_t s) {
  launch_k(k_seg_cycle_init, 1, 256, 0, s, st, ctl, relative_to_beta, cond);
  count_launches(1);
}

template <typename V>
void launch_seg_scale(JVec<V> x, const TileList& tl, const SegState* st, cudaStream_t s) {
  launch_k(k_seg_scale<V>, tl.ntiles, kKB, 0, s, x, tl.tiles, st);
  count_launches(1);
}
template void launch_seg_scale<double>(JVec<double>, const TileList&, const SegState*,
                                       cudaStream_t);
template void launch_seg_scale<float>(JVec<float>, const TileList&, const SegState*,
                                      cudaStream_t);

template <typename V, typename X>
void launch_seg_update_x(const SegState* st, const KCtl* ctl, const V* Z, int64_t n,
                         const TileList& tl, X* x, cudaStream_t s) {
  launch_k(k_seg_update_x<V, X>, tl.ntiles, kKB, 0, s, st, ctl, Z, n, tl.tiles, x);
  count_launches(1);
}
template void launch_seg_update_x<double, double>(const SegState*, const KCtl*, const double*,
                                                  int64_t, const TileList&, double*,
                                                  cudaStream_t);
template void launch_seg_update_x<float, float>(const SegState*, const KCtl*, const float*,
                                                int64_t, const TileList&, float*, cudaStream_t);

template <typename A, typename B>
void launch_seg_normalise(const A* in, B* out, const TileList& tl, const SegState* st,
                          cudaStream_t s) {
  launch_k(k_seg_normalise<A, B>, tl.ntiles, kKB, 0, s, in, out, tl.tiles, st);
  count_launches(1);
}
template void launch_seg_normalise<double, float>(const double*, float*, const TileList&,
                                                  const SegState*, cudaStream_t);

template <typename V, typename X>
void launch_seg_axpy(X* x, const V* d, const TileList& tl, const SegState* st, cudaStream_t s) {
  launch_k(k_seg_axpy<V, X>, tl.ntiles, kKB, 0, s, x, d, tl.tiles, st);
  count_launches(1);
}
template void launch_seg_axpy<float, double>(double*, const float*, const TileList&,
                                             const SegState*, cudaStream_t);

}  // namespace fs
