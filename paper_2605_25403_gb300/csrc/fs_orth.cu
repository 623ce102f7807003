// Orthogonalisation of the new Arnoldi vector of flexible GMRES(m) (paper
// Sec. 3.2, GMRES) and the Givens step of its Hessenberg column, in one
// cooperative launch on sm_103a.
//
// w = V[j+1] is orthogonalised against V[0..j], j = ctl->j, by classical
// Gram-Schmidt with the basis' own Gram matrix as the correction (the
// one-synchronisation CGS2 of Swirydowicz, Langou, Ananthan, Yang and Thomas,
// "Low synchronization Gram-Schmidt and GMRES algorithms", Numer. Linear
// Algebra Appl. 28, 2021):
//   dot: a = V^T w, e = V^T v_j - delta (the new row of E = V^T V - I),
//        ww = w.w
//   upd: h = a - E a  (what a second Gram-Schmidt pass would subtract:
//        V^T (w - V a) = -E a), hn^2 = ww - a.h, V[j+1] = (w - V h) / hn
// so the basis is read twice, where dot, update with re-dot and final update
// as separate passes read it four times.  When the subtraction cancels most
// of w (hn^2 < kRedo ww: the Pythagorean norm would lose digits) the update
// pass stores w' = w - V h with its re-dots, and a real second pass ends the
// step: h2 = V^T w', V[j+1] = (w' - V h2) / hn, hn^2 = ||w'||^2 - ||h2||^2.
// E comes from dot products of the stored vectors, so the correction keeps
// the loss of orthogonality from growing from step to step (plain one-pass
// Gram-Schmidt multiplies it by |h| / hn, about 3, at every step).  Its
// diagonal also gives the stored vectors' norms, one step late, to the least-
// squares problem (givens_warp): the Pythagorean norm has lost the digits that
// cancelled.
//
// Against two full passes, over chains of 30 steps: |V^T V - I| is 1e-7 in FP32
// and 1e-15 in FP64 with either when half of w^2 is new at every step; when 2%
// of it is, 1e-7 and 9e-16 with two passes, 3e-6 and 2e-14 with this one, all of
// it on the diagonal, which the rotations account for.
//
// Time per Arnoldi step inside the restart loop on GB300 (from the end of the
// product to the end of the step, Givens rotations included), as three
// kernels (dot, update with re-dot and Givens step, final update: the last
// block of each reduced the sums, one thread ran the rotations through global
// memory) and as this one launch:
//   8x8 square, FP64, 659 entries             65 us -> 18 us
//   256x48 channel, FP64, 112,115             71 us -> 28 us
//   512x96 channel, FP32, 445,411             46 us -> 22 us
//   48^3 cube, FP32, 2.86 million            153 us -> 84 us
//   96 squares, FP32, 4 million              103 us -> 90 us
// and per pass of the timing cases 1.03x (the batch) to 2.09x (the square).
//
// Two kernels share the arithmetic:
//   k_orth_one   one segment of up to kStreamShare entries per SM; bound by
//                latency (barrier, partial sums, one load round trip per
//                batch of basis vectors).  One grid barrier; every block
//                reduces the partial sums itself, in the same fixed order.
//   k_orth_many  batches, and single problems with more entries; bound by the
//                reads of the basis.  One block reduces a segment's sums
//                between two grid barriers.  FP32 vectors stream through
//                shared memory by TMA bulk copies, kept 192 KB ahead.
// A lane sums the products of its four entries of a chunk in the vector type, a
// warp adds them by a reduce-scatter in the vector type (128 products), chunks,
// warps and blocks are added in FP64.
// FP64 arithmetic runs at 1/58 of the FP32 rate on GB300 (one FP64 warp
// instruction takes 64 cycles of its quarter SM), so the scalar chains
// (square roots, quotients, rotations) are kept short and spread over lanes.
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "fs_device.h"

namespace fs {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kOrthWarps = 16;
constexpr int kOrthMain = 32 * kOrthWarps;       // threads that work on entries
constexpr int kOneThreads = kOrthMain + 32;      // k_orth_one: and a Givens warp
constexpr int kManyThreads = kOrthMain + 64;     // k_orth_many: a copying and a Givens warp
constexpr double kRedo = 0.01;
// j + 1 <= 31 basis vectors beside w: 2 (j + 1) + 1 sums in slots of 64, and
// lanes 30 and 31 of the ring's sums hold a_j and w.w
static_assert(kMaxRestart <= 31, "a lane per basis vector, 64 sums per slot");

template <typename V>
__device__ __forceinline__ V warp_sum(V v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
  return v;
}

__device__ __forceinline__ void main_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }

// 1 / sqrt(x) in FP64: the FP32 value and two Newton steps (relative error
// 1e-7, 2e-14, then rounding); x outside the FP32 range or not positive by
// the library's square root.
__device__ __forceinline__ double inv_sqrt(double x) {
  if (!(x > 1e-30 && x < 1e30)) return 1.0 / sqrt(x);
  double y = (double)rsqrtf((float)x);
  const double h = 0.5 * x;
  y = y * (1.5 - h * y * y);
  return y * (1.5 - h * y * y);
}

// A wait ran out: the cycle of every segment ends and the solve reports it
// (one thread).  Another block that did pass may be between its read of
// all_done and its own setting of the loop's condition (end_arnoldi_step), so
// the condition can end up set: the next pass then finds every segment done
// and clears it (end_loop).
__device__ void orth_give_up(SegState* st, KCtl* ctl, int nseg, cudaGraphConditionalHandle cond) {
  for (int s = 0; s < nseg; ++s) {
    st[s].bad = 2;
    st[s].done = 1;
  }
  ctl->all_done = 1;
  if (cond) cudaGraphSetConditional(cond, 0);
}

// Nothing left to do at a launch's start: the loop node (if any) ends here,
// whatever its condition was left at.
__device__ __forceinline__ void end_loop(cudaGraphConditionalHandle cond) {
  if (cond && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(cond, 0);
}

// Reduce-scatter of NB per-lane values over a warp (NB a power of two):
// at the level with xor offset o, a lane keeps half of its slots (the upper
// half when bit o of its index is set) and adds the partner's copy of them,
// so after log2(NB) levels lane l holds slot l / (32 / NB) summed over the
// lanes that share it, and the remaining levels finish that sum.  NB - 1 +
// 5 - log2(NB) additions per lane instead of 5 NB for NB separate sums.
template <int NB, typename R>
__device__ __forceinline__ R warp_transpose_sum(R (&v)[NB]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int half = NB / 2, off = 16; half >= 1; half /= 2, off /= 2) {
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const R send = hi ? v[i] : v[i + half];
      const R keep = hi ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(kFull, send, off);
    }
  }
  R s = v[0];
#pragma unroll
  for (int off = 16 / NB; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off);
  return s;
}

// The thread's entries e0 + T k, k < LE, of one vector (0 past len; full: no
// entry of the thread is).
template <typename V, int LE>
__device__ __forceinline__ void lane_load(const V* p, int e0, int T, int len, bool full,
                                          V (&x)[LE]) {
  if (full) {
#pragma unroll
    for (int k = 0; k < LE; ++k) x[k] = p[e0 + T * k];
  } else {
#pragma unroll
    for (int k = 0; k < LE; ++k) x[k] = e0 + T * k < len ? p[e0 + T * k] : V(0);
  }
}

// Dot products of a piece (len entries) with the basis vectors 0 .. nvec - 1
// (ld apart from base on): part[v] += v . y, with TWO part[nvec + v] += v . z,
// and after them += y . y.  T threads per group; the groups share the
// vectors, NB at a time.  FP32 sums run over the 128 products of a warp's
// chunk and are added in FP64; FP64 ones are taken across the warp once per
// batch.
template <typename V, int LE, int NB, bool TWO>
__device__ __forceinline__ void dot_piece(const V* base, int64_t ld, int nvec, const V* y,
                                          const V* z, int len, int T, double* part) {
  constexpr bool f32 = sizeof(V) == 4;
  static_assert(!f32 || LE <= 4, "FP32 sums of at most 128 products");
  static_assert(32 / NB >= 4, "three lanes of a slot");
  const int lane = threadIdx.x & 31, NG = kOrthMain / T;
  const int grp = threadIdx.x / T, t = threadIdx.x - grp * T;
  for (int v0 = grp * NB; v0 < nvec; v0 += NG * NB) {
    const int nb = min(NB, nvec - v0);
    const V* bv = base + (int64_t)v0 * ld;
    V d[NB], e[NB], yy = V(0);
#pragma unroll
    for (int b = 0; b < NB; ++b) d[b] = e[b] = V(0);
    // the warp's sums: of v . y, v . z and y . y in a slot's first three lanes,
    // so that one FP64 instruction adds all of them
    constexpr int kShare = 32 / NB;  // lanes holding one slot's sum
    const int slot = lane / kShare, which = lane % kShare;
    double acc = 0;
    auto take = [&]() {
      const V sd = warp_transpose_sum<NB, V>(d);
      V se = V(0), sy = V(0);
      if constexpr (TWO) se = warp_transpose_sum<NB, V>(e);
      if (v0 == 0) sy = warp_sum(yy);
      acc += (double)(which == 0 ? sd : which == 1 ? se : sy);
    };
    for (int c0 = 0; c0 + (t & ~31) < len; c0 += T * LE) {
      const int e0 = c0 + t;
      const bool full = c0 + T * LE <= len;
      V w[LE], u[LE], x[NB][LE];
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (b < nb) lane_load<V, LE>(bv + (int64_t)b * ld, e0, T, len, full, x[b]);
      lane_load<V, LE>(y, e0, T, len, full, w);
      if constexpr (TWO) lane_load<V, LE>(z, e0, T, len, full, u);
      if constexpr (f32) {
        yy = V(0);
#pragma unroll
        for (int b = 0; b < NB; ++b) d[b] = e[b] = V(0);
      }
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (b < nb) {
#pragma unroll
          for (int k = 0; k < LE; ++k) {
            d[b] += x[b][k] * w[k];
            if constexpr (TWO) e[b] += x[b][k] * u[k];
          }
        }
      if (v0 == 0) {
#pragma unroll
        for (int k = 0; k < LE; ++k) yy += w[k] * w[k];
      }
      if constexpr (f32) take();
    }
    if constexpr (!f32) take();
    if (which < (TWO ? 2 : 1) && slot < nb) part[which * nvec + v0 + slot] += acc;
    if (v0 == 0 && lane == 2) part[TWO ? 2 * nvec : nvec] += acc;
  }
}

// w = (w - sum_v coef[v] v) f over a piece.
template <typename V, int LU, int NB>
__device__ __forceinline__ void upd_piece(const V* base, int64_t ld, int nvec, V* w, int len,
                                          const V* coef, V f) {
  const int t = threadIdx.x;
  for (int c0 = 0; c0 + (t & ~31) < len; c0 += kOrthMain * LU) {
    const int e0 = c0 + t;
    const bool full = c0 + kOrthMain * LU <= len;
    V x[LU], acc[LU];
    lane_load<V, LU>(w, e0, kOrthMain, len, full, x);
#pragma unroll
    for (int k = 0; k < LU; ++k) acc[k] = V(0);
    for (int v0 = 0; v0 < nvec; v0 += NB) {
      const int nb = min(NB, nvec - v0);
      const V* bv = base + (int64_t)v0 * ld;
      V y[NB][LU];
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (b < nb) lane_load<V, LU>(bv + (int64_t)b * ld, e0, kOrthMain, len, full, y[b]);
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (b < nb) {
          const V c = coef[v0 + b];
#pragma unroll
          for (int k = 0; k < LU; ++k) acc[k] += c * y[b][k];
        }
    }
#pragma unroll
    for (int k = 0; k < LU; ++k)
      if (full || e0 + kOrthMain * k < len) w[e0 + kOrthMain * k] = (x[k] - acc[k]) * f;
  }
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* b, unsigned count) {
  asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(smem_addr(b)), "r"(bytes)
               : "memory");
}
// Waits for the phase with the given parity; false after `limit` nanoseconds.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, unsigned parity, uint64_t limit) {
  const uint32_t a = smem_addr(b);
  uint64_t t0 = 0;
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    const uint64_t t = now_ns();
    if (!t0) t0 = t;
    if (t - t0 >= limit) return false;
  }
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// A segment's E, held in the type of its vectors.
template <typename V>
__host__ __device__ __forceinline__ V* gram(SegState& S) {
  return reinterpret_cast<V*>(S.E);
}

// Its rows and columns below j into shared memory (one warp; the loads eight at
// a time: one by one they outlast the dot pass of a small problem).
template <typename V>
__device__ __forceinline__ void load_gram(V* dst, const V* src, int j) {
  const int lane = threadIdx.x & 31;
  for (int i = 0; i < j; i += 8) {
    V v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = i + u < j && lane < j ? src[(i + u) * 32 + lane] : V(0);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i + u < j) dst[(i + u) * 33 + lane] = v[u];
  }
}

// Shared by both kernels.
template <typename V>
struct OrthShared {
  double wpart[kOrthWarps][64];  // a warp's sums
  double red[kOrthMain];
  double sum[64];
  V vsum[64];  // the first reduction's in the vectors' type, e_j less its 1
  double hcol[kMaxRestart + 1];  // the Hessenberg column
  V E[32 * 33];
  V c[4][32];  // E a (FP64: in four shares of the columns)
  double f;    // 1 / hn
  int redo, ok;
};

template <typename V>
__device__ __forceinline__ void clear_sums(OrthShared<V>& sh, int ns) {
  for (int i = threadIdx.x; i < kOrthWarps * 64; i += blockDim.x)
    if ((i & 63) < ns) (&sh.wpart[0][0])[i] = 0.0;
}
// A slot's first ns sums from the warps' (threads 0 .. ns - 1).
template <typename V>
__device__ __forceinline__ void store_sums(const OrthShared<V>& sh, double* slot, int ns) {
  if (threadIdx.x < ns) {
    double s[4] = {0, 0, 0, 0};
#pragma unroll
    for (int w = 0; w < kOrthWarps; ++w) s[w & 3] += sh.wpart[w][threadIdx.x];
    slot[threadIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
  }
}

// sh.sum = the first ns sums added over count slots (64 apart), in a fixed
// order (whole block).  unit: the index of v_j . v_j among them (-1: none).
template <typename V>
__device__ __forceinline__ void reduce_sums(OrthShared<V>& sh, const double* part, int ns,
                                            int count, int unit) {
  const int tid = threadIdx.x;
  const int parts = kOrthMain / ns, g = tid / ns, s = tid - g * ns;
  if (g < parts) {
    double acc[4] = {0, 0, 0, 0};
    const double* q = part + s;
    int k = g;
    for (; k + 3 * parts < count; k += 4 * parts) {
      double v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = __ldcg(q + (int64_t)(k + u * parts) * 64);
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] += v[u];
    }
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (k + u * parts < count) acc[u] += __ldcg(q + (int64_t)(k + u * parts) * 64);
    sh.red[tid] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  }
  __syncthreads();
  if (tid < ns) {
    double v[4] = {0, 0, 0, 0};
    const int used = parts < count ? parts : count;
    for (int q = 0; q < used; q += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (q + u < used) v[u] += sh.red[(q + u) * ns + tid];
    }
    const double s = (v[0] + v[1]) + (v[2] + v[3]);
    sh.sum[tid] = s;
    if (unit >= 0) sh.vsum[tid] = (V)(tid == unit ? s - 1.0 : s);
  }
  __syncthreads();
}

// What a launch runs: a whole Arnoldi step with its Givens rotations, or
// for timing the orthogonalisation alone, with both passes taken (ORTH_FULL),
// with the first only (ORTH_ONCE), or one of its passes.
enum { ORTH_STEP = 0, ORTH_FULL, ORTH_ONCE, ORTH_DOT, ORTH_UPD, ORTH_FIN };
__device__ __forceinline__ bool second_pass(int mode, double hn2, double ww) {
  return mode == ORTH_STEP ? hn2 < kRedo * ww : mode != ORTH_ONCE;
}

// From the sums of the dot pass (sh.sum) and E: c = E a, then h, hn and the
// decision on a second pass (whole block; sh.hcol, sh.f and sh.redo are
// valid after the caller's next barrier).  Row j of E goes to S when store.
// In FP32 a warp takes a row of E a and adds it over its lanes; in FP64,
// whose additions over the lanes would cost most of it, a lane takes a row
// and four warps (one per quarter SM) eight columns each.
template <typename V>
__device__ __forceinline__ void first_column(OrthShared<V>& sh, int j, int mode, SegState& S,
                                             bool store) {
  constexpr bool f32 = sizeof(V) == 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nvec = j + 1;
  const V e = lane < nvec ? sh.vsum[nvec + lane] : V(0);
  if (f32 && warp < kOrthWarps) {
    const V a = lane < nvec ? sh.vsum[lane] : V(0);
    for (int i = warp; i < nvec; i += kOrthWarps) {
      // row i of E: E[i][k] for k < j, e_i in column j; row j is e
      const V ei = __shfl_sync(kFull, e, i);
      const V r = i == j ? e : lane < j ? sh.E[i * 33 + lane] : lane == j ? ei : V(0);
      const V s = warp_sum(r * a);
      if (lane == 0) sh.c[0][i] = s;
    }
  } else if (!f32 && warp < 4) {
    V s = V(0);
    for (int k = 8 * warp; k < 8 * warp + 8 && k < nvec; ++k) {
      const V ek = __shfl_sync(kFull, e, k);
      const V r = lane == j ? ek : lane > j ? V(0) : k == j ? e : sh.E[lane * 33 + k];
      s += r * sh.vsum[k];
    }
    sh.c[warp][lane] = s;
  } else if (warp >= kOrthWarps && store && lane < nvec) {
    gram<V>(S)[lane * 32 + j] = e;
    gram<V>(S)[j * 32 + lane] = e;
  }
  __syncthreads();
  if (warp == 0) {
    const double ad = lane < nvec ? sh.sum[lane] : 0.0;
    double c = (double)sh.c[0][lane];
    if constexpr (!f32) c = (c + sh.c[1][lane]) + (sh.c[2][lane] + sh.c[3][lane]);
    const double h = lane < nvec ? ad - c : 0.0;
    const double ww = sh.sum[2 * nvec];
    const double hn2 = ww - warp_sum(ad * h);
    const double f = inv_sqrt(fmax(hn2, 0.0));
    if (lane < nvec) sh.hcol[lane] = h;
    if (lane == 0) {
      sh.hcol[nvec] = hn2 > 0.0 ? hn2 * f : isfinite(hn2) ? 0.0 : hn2;
      sh.f = f;
      sh.redo = second_pass(mode, hn2, ww) ? 1 : 0;
    }
  }
}

// After the second pass' sums: h2, and the column with hfirst (warp 0).
template <typename V>
__device__ __forceinline__ void second_column(OrthShared<V>& sh, int nvec, const double* hfirst) {
  const int lane = threadIdx.x & 31;
  const double h2 = lane < nvec ? sh.sum[lane] : 0.0;
  const double hn2 = sh.sum[nvec] - warp_sum(h2 * h2);
  const double f = inv_sqrt(fmax(hn2, 0.0));
  if (lane < nvec) sh.hcol[lane] = hfirst[lane] + h2;
  if (lane == 0) {
    sh.hcol[nvec] = hn2 > 0.0 ? hn2 * f : isfinite(hn2) ? 0.0 : hn2;
    sh.f = f;
  }
}

// Givens rotations of column j of one active segment's Hessenberg matrix
// (col[0..j+1]), its least-squares residual, and the end of its cycle
// (converged, broken or at the restart length): the segment is then marked
// done and counted.  One warp: a lane holds a rotation and its operand, so
// the chain of rotations is one FMA per step.
//
// The least-squares problem is that of the unit vectors v_l / |v_l|.  The norm
// by Pythagoras, ww - a.h, has lost the digits that cancel (FP32, hn^2 at 2%
// of ww: 3e-6 of the norm, where the sums themselves carry 1e-7), but one step
// later the dot pass finds |v_j|^2 itself, the diagonal of E.  So the rows of
// the column are scaled by |v_l|, and the entry below the diagonal of the
// column before, hn |v_j|, and its rotation are brought up to date first.
// x: the lane's |v_l|^2 - 1.  The rotation's update is a correction of rounding
// size, relative to what it corrects, so FP32 holds it; its operands are read
// with the others and its arithmetic runs beside the chain of rotations, which
// is the launch's critical path on small problems.
template <typename V>
__device__ void givens_warp(SegState& S, KCtl* ctl, int j, int m, const double* col, V x) {
  const int lane = threadIdx.x & 31, p = j > 0 ? j - 1 : 0;
  double cs = lane < j ? S.cs[lane] : 1.0, sn = lane < j ? S.sn[lane] : 0.0;
  double gj = S.g[j], gp = S.g[p], hp = S.H[p * m + p];
  const double tol = S.tol_abs;
  const V off = lane <= j ? x * (V(0.5) - V(0.125) * x) : V(0);  // |v_l| - 1
  const double h = lane <= j + 1 ? col[lane] : 0.0, hl = h + h * (double)off;
  // b -> b (1 + d) in the rotation before: den^2 = a^2 + b^2 grows by 1 + 2 q
  const float d = (float)__shfl_sync(kFull, off, j), s0 = __shfl_sync(kFull, (float)sn, p);
  const float q = s0 * s0 * (d + 0.5f * d * d), r = q * (1.5f * q - 1.0f);  // 1/sqrt(1+2q) - 1
  const double dc = (double)r, ds = (double)(d + r + d * r);
  // the entry below the diagonal of rotation l, and the one it starts from
  const double b = __shfl_down_sync(kFull, hl, 1);
  double cb = cs * b;
  double a = __shfl_sync(kFull, hl, 0), mine = a;
  for (int i = 0; i < j - 1; ++i) {
    a = fma(-__shfl_sync(kFull, sn, i), a, __shfl_sync(kFull, cb, i));
    if (lane == i + 1) mine = a;
  }
  if (j > 0) {
    if (lane == p) {
      cs += cs * dc;
      sn += sn * ds;
      cb = cs * b;
      S.cs[p] = cs;
      S.sn[p] = sn;
    }
    gj += gj * ds;
    a = fma(-__shfl_sync(kFull, sn, p), a, __shfl_sync(kFull, cb, p));
    if (lane == j) mine = a;
    if (lane == 0) {
      S.g[p] = gp + gp * dc;
      S.H[p * m + p] = hp + hp * (double)(q - 0.5f * q * q);
    }
  }
  const double bl = __shfl_sync(kFull, b, j);
  // the new rotation: c = a / den, s = b / den, den = sqrt(a^2 + b^2), the
  // pair scaled by its larger entry
  const double big = fmax(fabs(a), fabs(bl));
  double c = 1.0, s = 0.0, den = big;
  if (big > 0.0) {
    const int ex = ilogb(big);
    const double as = scalbn(a, -ex), bs = scalbn(bl, -ex);
    const double r2 = as * as + bs * bs, ri = inv_sqrt(r2);
    c = as * ri;
    s = bs * ri;
    den = scalbn(r2 * ri, ex);
  }
  if (!isfinite(a) || !isfinite(bl)) den = a + bl + INFINITY;
  const double out = lane < j ? cs * mine + sn * b : lane == j ? den : 0.0;
  if (lane <= j + 1) S.H[lane * m + j] = out;
  if (lane == 0) {
    S.cs[j] = c;
    S.sn[j] = s;
    S.g[j + 1] = -s * gj;
    S.g[j] = c * gj;
    const double resid = fabs(s * gj);
    S.resid = resid;
    S.k = j + 1;
    bool finish = false;
    if (!isfinite(resid) || !isfinite(den) || den == 0.0) {
      S.bad = isfinite(resid) && isfinite(den) ? S.bad : 1;
      S.k = j;  // drop the broken column
      finish = true;
    } else if (resid <= tol || bl == 0.0 || j + 1 >= m) {
      finish = true;
    }
    if (finish) {
      S.done = 1;
      if (atomicAdd(&ctl->ndone, 1) + 1 == ctl->nseg) ctl->all_done = 1;
    }
  }
}

// The step index advances and the loop node's condition (if any) becomes
// "a segment is still active and j + 1 < m" (one thread).
__device__ void end_arnoldi_step(KCtl* ctl, int j, int m, cudaGraphConditionalHandle cond) {
  const int all = atomicAdd(&ctl->all_done, 0);
  ctl->j = j + 1;
  if (cond) cudaGraphSetConditional(cond, (!all && j + 1 < m) ? 1u : 0u);
}

// ---------------------------------------------------------------------------
// One segment, share entries per block from block b's b share on.  (Keeping
// the block's share of the basis in shared memory between the passes, by bulk
// copies issued at the start, measured no faster: the update pass re-reads
// it from L1 and L2 as quickly, and the copies start later than the loads.)
// ---------------------------------------------------------------------------
template <typename V, int LU>
__global__ void __launch_bounds__(kOneThreads, 1)
    k_orth_one(V* Vb, int64_t ld, OrthPlan P, SegState* st, KCtl* ctl,
               cudaGraphConditionalHandle cond, int mode) {
  // dot pass: NB vectors of LE entries per thread at a time; update: NBU of LU
  constexpr bool f32 = sizeof(V) == 4;
  constexpr int LE = 4, NB = f32 ? 8 : 2;
  constexpr int NBU = f32 ? (LU == 4 ? 8 : 16) : 8;
  __shared__ OrthShared<V> sh;
  __shared__ V coef[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool work = warp < kOrthWarps;
  SegState& S = st[0];
  const int j = ctl->j, m = ctl->m, nvec = j + 1;
  const unsigned base = ctl->bar_base;
  const uint64_t limit = ctl->wait_ns;  // of each wait
  if (mode == ORTH_STEP && S.done) return end_loop(cond);
  const int n1 = 2 * nvec + 1, n2 = nvec + 1;  // sums of the first and second reduction
  const int64_t start = (int64_t)blockIdx.x * P.share;
  const int len = (int)(P.n - start < P.share ? P.n - start : P.share);
  const bool owner = blockIdx.x == 0;
  double* part1 = P.partial;
  double* part2 = P.partial + (int64_t)gridDim.x * 64;
  V* bv = Vb + start;
  V* vw = bv + (int64_t)nvec * ld;
  clear_sums(sh, n1);
  if (mode == ORTH_UPD && !work)
    for (int i = 0; i < 33; ++i) sh.E[i * 32 + lane] = V(0);
  __syncthreads();
  if (mode <= ORTH_DOT) {
    if (work)
      dot_piece<V, LE, NB, true>(bv, ld, nvec, vw, vw - ld, len, P.T, sh.wpart[warp]);
    else if (mode < ORTH_DOT)
      load_gram(sh.E, gram<V>(S), j);  // while the dot pass runs
    __syncthreads();
    store_sums(sh, part1 + (int64_t)blockIdx.x * 64, n1);
    if (mode == ORTH_DOT) return;
  }
  unsigned bars = 0;
  if (mode < ORTH_DOT) {
    bars += 1;
    if (!grid_barrier(&ctl->bar, base + bars * gridDim.x, limit, &sh.ok)) {
      if (tid == 0) orth_give_up(st, ctl, 1, cond);
      return;
    }
  }
  bool redo = true;
  V vsq = V(0);  // |v_lane|^2 - 1
  if (mode != ORTH_FIN) {
    reduce_sums(sh, part1, n1, gridDim.x, nvec + j);
    clear_sums(sh, n2);
    first_column(sh, j, mode, S, owner && mode == ORTH_STEP);
    __syncthreads();
    redo = sh.redo != 0;
    if (!work && lane <= j)
      vsq = lane < j ? sh.E[lane * 34] : sh.vsum[nvec + j];
    if (work && lane < nvec) coef[lane] = (V)sh.hcol[lane];  // every warp the same values
    if (!work && owner && mode == ORTH_STEP) {
      if (!redo) {
        givens_warp(S, ctl, j, m, sh.hcol, vsq);
        if (lane == 0) end_arnoldi_step(ctl, j, m, cond);
      } else if (lane < nvec) {
        S.h2[lane] = sh.hcol[lane];  // the first pass' share of the column
      }
    }
    if (work) {
      __syncwarp();
      upd_piece<V, LU, NBU>(bv, ld, nvec, vw, len, coef, redo ? V(1) : (V)sh.f);
    }
    if (redo) {  // the dots of w', which other threads of the block wrote
      __syncthreads();
      if (work)
        dot_piece<V, LE, NB, false>(bv, ld, nvec, vw, nullptr, len, P.T, sh.wpart[warp]);
      __syncthreads();
      store_sums(sh, part2 + (int64_t)blockIdx.x * 64, n2);
    }
    if (mode == ORTH_UPD) return;
    // second pass: every block took the same decision
    if (redo) {
      bars += 1;
      if (!grid_barrier(&ctl->bar, base + bars * gridDim.x, limit, &sh.ok)) {
        if (tid == 0) orth_give_up(st, ctl, 1, cond);
        return;
      }
    }
  }
  if (owner && tid == 0) ctl->bar_base = base + bars * gridDim.x;
  if (!redo) return;
  reduce_sums(sh, part2, n2, gridDim.x, -1);
  if (warp == 0) second_column(sh, nvec, S.h2);
  __syncthreads();
  if (work && lane < nvec) coef[lane] = (V)sh.sum[lane];
  if (!work && owner && mode == ORTH_STEP) {
    givens_warp(S, ctl, j, m, sh.hcol, vsq);
    if (lane == 0) end_arnoldi_step(ctl, j, m, cond);
  }
  if (work) {
    __syncwarp();
    upd_piece<V, LU, NBU>(bv, ld, nvec, vw, len, coef, (V)sh.f);
  }
}

// ---------------------------------------------------------------------------
// Batches and large vectors.  Pieces of one segment each are dealt to the
// blocks in turn, so that the pieces of the segments still active spread over
// the chip; a block's pieces of one segment share a slot of partial sums.
// After the dot pass and a barrier, block s mod gridDim reduces segment s and
// writes its coefficients to the segment state; after a second barrier every
// block updates its pieces, while a warp of the reducing block takes the
// Givens step.
// ---------------------------------------------------------------------------
// The FP32 ring: stages of kGV vectors x kChunk entries, filled by bulk
// copies that the 17th warp issues, emptied by the 16 others.
constexpr int kChunk = kOrthPiece;
static_assert(kChunk == kOrthMain * 4, "a float4 per thread");
constexpr int kGV = 4;
constexpr int kStages = 6;
constexpr size_t kRingBytes = (size_t)kStages * kGV * kChunk * sizeof(float);

struct Ring {
  uint64_t full[kStages], empty[kStages];
  uint64_t limit;  // of each wait, ns
};

// Of kOrthList pieces of the block, those whose segment takes part, in order.
struct PieceList {
  int32_t p[kOrthList];
  int32_t count, warps[kManyThreads / 32];
};

// Fills the list from the block's pieces r kOrthList on (whole block): a
// thread looks at a piece, warps place theirs by a ballot.
template <typename F>
__device__ __forceinline__ void list_pieces(PieceList& L, int npiece, int r, F takes_part) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, G = gridDim.x;
  int done = 0;
  __syncthreads();
  for (int k0 = r * kOrthList;
       k0 < (r + 1) * kOrthList && blockIdx.x + (int64_t)k0 * G < npiece; k0 += kManyThreads) {
    const int64_t p = blockIdx.x + (int64_t)(k0 + tid) * G;
    const bool in = k0 + tid < (r + 1) * kOrthList && p < npiece && takes_part((int)p);
    const unsigned all = __ballot_sync(kFull, in);
    if (lane == 0) L.warps[warp] = __popc(all);
    __syncthreads();
    int at = done, sum = done;
    for (int w = 0; w < kManyThreads / 32; ++w) {
      if (w == warp) at = sum;
      sum += L.warps[w];
    }
    if (in) L.p[at + __popc(all & ((1u << lane) - 1))] = (int32_t)p;
    done = sum;
    __syncthreads();
  }
  if (tid == 0) L.count = done;
  __syncthreads();
}

// Chunk c0 of a piece whose first entry is head entries behind a 16-byte
// boundary: floats copied per vector (a multiple of 4; the rows of the basis
// are padded to one).
__device__ __forceinline__ int chunk_floats(int c0, int head, int len) {
  const int rest = head + len - c0;
  return rest >= kChunk ? kChunk : (rest + 3) & ~3;
}

// Producer (one lane): the vectors `first` (basis index), then `second` when
// not negative, then 0 .. nrest - 1, chunk by chunk.  it counts the stages
// filled since the kernel's start.
__device__ __forceinline__ bool ring_fill(const float* Vb, int64_t ld, int64_t start, int len,
                                          int first, int second, int nrest, float* ring, Ring& R,
                                          unsigned& it) {
  const int head = (int)(start & 3), lead = second < 0 ? 1 : 2, nseq = lead + nrest;
  const float* src = Vb + (start - head);
  for (int c0 = 0; c0 < head + len; c0 += kChunk) {
    const unsigned bytes = 4u * chunk_floats(c0, head, len);
    for (int q = 0; q < nseq; q += kGV) {
      const unsigned s = it % kStages, use = it / kStages;
      if (use > 0 && !mbar_wait(&R.empty[s], (use - 1) & 1, R.limit)) return false;
      const int nv = min(kGV, nseq - q);
      mbar_expect(&R.full[s], bytes * nv);
      for (int k = 0; k < nv; ++k) {
        const int i = q + k;
        const int v = i == 0 ? first : (i == 1 && lead == 2) ? second : i - lead;
        bulk_copy(ring + ((size_t)s * kGV + k) * kChunk, src + (int64_t)v * ld + c0, bytes,
                  &R.full[s]);
      }
      ++it;
    }
  }
  return true;
}

// Entries 4 t .. 4 t + 3 of a ring vector, with those outside [lo, hi) zero.
__device__ __forceinline__ void ring_get(const float* p, int t, bool all, int lo, int hi,
                                         float (&x)[4]) {
  const float4 q = reinterpret_cast<const float4*>(p)[t];
  x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
  if (!all) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (4 * t + k < lo || 4 * t + k >= hi) x[k] = 0.0f;
  }
}

// Dot pass of one piece from the ring (order: w, v_j, v_0 .. v_{j-1}); the
// lane's FP64 sums: sa of a_lane (lane 30: a_j, lane 31: ww), se of e_lane
// (lane 30: e_j + 1).  FP32 sums run over at most 128 products.
__device__ __forceinline__ void ring_dot(const float* ring, Ring& R, unsigned& it, bool& ok,
                                         int head, int len, int j, double& sa, double& se) {
  const int t = threadIdx.x, lane = t & 31, nseq = j + 2;
  for (int c0 = 0; c0 < head + len; c0 += kChunk) {
    const int lo = head - c0, hi = head + len - c0;
    const bool all = lo <= 0 && hi >= kChunk;
    float d[32], e[32], w[4], u[4];
#pragma unroll
    for (int i = 0; i < 32; ++i) d[i] = e[i] = 0.0f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (kGV * q < nseq) {
        const unsigned s = it % kStages;
        ok = ok && mbar_wait(&R.full[s], (it / kStages) & 1, R.limit);
        const float* p = ring + (size_t)s * kGV * kChunk;
#pragma unroll
        for (int k = 0; k < kGV; ++k) {
          const int i = kGV * q + k;
          if (i < nseq) {
            float x[4];
            ring_get(p + k * kChunk, t, all, lo, hi, x);
            if (i == 0) {
#pragma unroll
              for (int b = 0; b < 4; ++b) {
                w[b] = x[b];
                d[31] += x[b] * x[b];
              }
            } else if (i == 1) {
#pragma unroll
              for (int b = 0; b < 4; ++b) {
                u[b] = x[b];
                d[30] += w[b] * x[b];
                e[30] += x[b] * x[b];
              }
            } else {
#pragma unroll
              for (int b = 0; b < 4; ++b) {
                d[i - 2] += x[b] * w[b];
                e[i - 2] += x[b] * u[b];
              }
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&R.empty[s]);
        ++it;
      }
    }
    sa += (double)warp_transpose_sum<32, float>(d);
    se += (double)warp_transpose_sum<32, float>(e);
  }
}

// Update pass of one piece from the ring (order: w, v_0 .. v_j).
__device__ __forceinline__ void ring_upd(const float* ring, Ring& R, unsigned& it, bool& ok,
                                         float* wp, int head, int len, int nvec,
                                         const float* coef, float f) {
  const int t = threadIdx.x, lane = t & 31, nseq = nvec + 1;
  float* out = wp - head;  // 16-byte boundary
  for (int c0 = 0; c0 < head + len; c0 += kChunk) {
    const int lo = head - c0, hi = head + len - c0;
    float acc[4];
    for (int q = 0; q < nseq; q += kGV) {
      const unsigned s = it % kStages;
      ok = ok && mbar_wait(&R.full[s], (it / kStages) & 1, R.limit);
      const float* p = ring + (size_t)s * kGV * kChunk;
#pragma unroll
      for (int k = 0; k < kGV; ++k) {
        const int i = q + k;
        if (i < nseq) {
          float x[4];
          ring_get(p + k * kChunk, t, true, 0, 0, x);
          const float c = i == 0 ? 0.0f : coef[i - 1];
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[b] = i == 0 ? x[b] : acc[b] - c * x[b];
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&R.empty[s]);
      ++it;
    }
    const int e0 = 4 * t;
    if (e0 >= lo && e0 + 4 <= hi) {
      *reinterpret_cast<float4*>(out + c0 + e0) =
          make_float4(acc[0] * f, acc[1] * f, acc[2] * f, acc[3] * f);
    } else {
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (e0 + b >= lo && e0 + b < hi) out[c0 + e0 + b] = acc[b] * f;
    }
  }
}

template <typename V>
__global__ void __launch_bounds__(kManyThreads, 1)
    k_orth_many(V* Vb, int64_t ld, OrthPlan P, SegState* st, KCtl* ctl,
                cudaGraphConditionalHandle cond, int mode) {
  constexpr bool f32 = sizeof(V) == 4;
  constexpr int LE = f32 ? 2 : 4, NB = f32 ? 8 : 2;
  extern __shared__ __align__(128) unsigned char smem[];
  float* ring = reinterpret_cast<float*>(smem);
  __shared__ OrthShared<V> sh;
  __shared__ Ring R;
  __shared__ PieceList L;
  __shared__ V coef[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, G = gridDim.x;
  const bool work = warp < kOrthWarps, copier = warp == kOrthWarps;
  const bool givens = warp == kOrthWarps + 1;
  const int j = ctl->j, m = ctl->m, nvec = j + 1, nseg = ctl->nseg;
  const unsigned base = ctl->bar_base;
  const uint64_t limit = ctl->wait_ns;  // of each wait
  if (mode == ORTH_STEP && ctl->all_done) return end_loop(cond);
  const int n1 = 2 * nvec + 1, n2 = nvec + 1;
  double* part1 = P.partial;
  double* part2 = P.partial + (int64_t)P.nslot * 64;
  unsigned it = 0;
  bool ok = true;
  if (f32 && tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&R.full[s], 1);
      mbar_init(&R.empty[s], kOrthWarps);
    }
    R.limit = limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  clear_sums(sh, n1);
  __syncthreads();
  // one round unless a block has more pieces than its list holds
  const int per = (P.npiece + G - 1) / G, rounds = (per + kOrthList - 1) / kOrthList;
  auto list_active = [&](int r) {  // at the kernel's start
    list_pieces(L, P.npiece, r, [&](int p) {
      return nseg == 1 || mode != ORTH_STEP || !st[P.pieces[p].seg].done;
    });
    return L.count;
  };
  auto list_again = [&](int r) {  // the same pieces, after the Givens steps
    if (rounds > 1)
      list_pieces(L, P.npiece, r, [&](int p) { return st[P.pieces[p].seg].act != 0; });
    return L.count;
  };
  if (mode > ORTH_DOT) list_active(0);

  // ---- dot pass -----------------------------------------------------------
  for (int r = 0; r < rounds && mode <= ORTH_DOT; ++r) {
    const int count = list_active(r);
    if (work && count > 0) {
      double sa = 0, se = 0;
      // a piece's record is read while the one before is worked on
      Tile qn = P.pieces[L.p[0]];
      int sn = P.slot[L.p[0]];
      for (int k = 0; k < count; ++k) {
        const Tile q = qn;
        const int slot = sn;
        if (k + 1 < count) {
          qn = P.pieces[L.p[k + 1]];
          sn = P.slot[L.p[k + 1]];
        } else {
          sn = -1;
        }
        if constexpr (f32) {
          ring_dot(ring, R, it, ok, (int)(q.start & 3), q.len, j, sa, se);
          if (sn != slot) {
            main_sync();  // the previous slot's sums are stored
            if (lane < j) {
              sh.wpart[warp][lane] = sa;
              sh.wpart[warp][nvec + lane] = se;
            } else if (lane == 30) {
              sh.wpart[warp][j] = sa;
              sh.wpart[warp][nvec + j] = se;
            } else if (lane == 31) {
              sh.wpart[warp][2 * nvec] = sa;
            }
            sa = se = 0;
            main_sync();
            store_sums(sh, part1 + (int64_t)slot * 64, n1);
          }
        } else {
          const V* vw = Vb + q.start + (int64_t)nvec * ld;
          dot_piece<V, LE, NB, true>(Vb + q.start, ld, nvec, vw, vw - ld, q.len, P.T,
                                     sh.wpart[warp]);
          if (sn != slot) {
            main_sync();
            store_sums(sh, part1 + (int64_t)slot * 64, n1);
            main_sync();
            for (int i = lane; i < n1; i += 32) sh.wpart[warp][i] = 0.0;
            __syncwarp();
          }
        }
      }
    } else if constexpr (f32) {
      if (copier && lane == 0)
        for (int k = 0; k < count && ok; ++k) {
          const Tile q = P.pieces[L.p[k]];
          ok = ring_fill(Vb, ld, q.start, q.len, nvec, j, j, ring, R, it);
        }
    }
  }
  // Before a block ends, its copies have landed.  They have when every wait
  // for a full stage ended; behind one that ran out, or a copying warp that
  // gave up, some may be under way, and the shared memory they write to
  // belongs to the next block.
  auto land = [&]() {
    if (f32 && copier && lane == 0)
      for (unsigned k = it > kStages ? it - kStages : 0; k < it; ++k)
        mbar_wait(&R.full[k % kStages], (k / kStages) & 1, kWaitNs);
  };
  if (mode == ORTH_DOT) return land();
  unsigned bars = 0;
  auto meet = [&]() {
    bars += 1;
    if (grid_barrier(&ctl->bar, base + bars * G, limit, &sh.ok)) return true;
    if (tid == 0) orth_give_up(st, ctl, nseg, cond);
    land();
    return false;
  };
  // the last segment handled ends the step (one thread)
  auto count_segment = [&]() {
    __threadfence();
    if (atomicAdd(&ctl->nfin, 1) == nseg - 1) {
      ctl->nfin = 0;
      __threadfence();
      end_arnoldi_step(ctl, j, m, cond);
    }
  };
  if (mode < ORTH_DOT && !meet()) return;

  // ---- columns of the segments ---------------------------------------------
  if (mode != ORTH_FIN) {
    for (int s = blockIdx.x; s < nseg; s += G) {
      SegState& S = st[s];
      __syncthreads();  // sh is free
      if (mode == ORTH_STEP && S.done) {
        if (tid == 0) S.act = 0;
        continue;
      }
      if (givens && mode == ORTH_STEP) load_gram(sh.E, gram<V>(S), j);
      if (givens && mode != ORTH_STEP)
        for (int i = 0; i < 33; ++i) sh.E[i * 32 + lane] = V(0);
      reduce_sums(sh, part1 + (int64_t)P.seg_slot[2 * s] * 64, n1, P.seg_slot[2 * s + 1],
                  nvec + j);
      first_column(sh, j, mode, S, mode == ORTH_STEP);
      __syncthreads();
      if (warp == 0) {
        if (lane <= nvec) S.h2[lane] = sh.hcol[lane];
        if (lane == 0) {
          S.f = sh.f;
          S.act = sh.redo ? 2 : 1;
          if (sh.redo) atomicAdd(&ctl->nredo, 1);
        }
      }
    }
    if (mode < ORTH_DOT && !meet()) return;

    // ---- update pass ------------------------------------------------------
    if (givens && mode == ORTH_STEP)
      for (int s = blockIdx.x; s < nseg; s += G) {
        SegState& S = st[s];
        const int act = S.act;
        if (act == 2) continue;
        if (act == 1) {
          if (lane <= nvec) sh.hcol[lane] = S.h2[lane];
          const V vsq = lane <= j ? gram<V>(S)[lane * 33] : V(0);
          __syncwarp();
          givens_warp(S, ctl, j, m, sh.hcol, vsq);
        }
        if (lane == 0) count_segment();
        __syncwarp();
      }
    for (int r = 0; r < rounds; ++r) {
      const int count = list_again(r);
      if (work && count > 0) {
        // records two pieces ahead, a segment's coefficients one ahead
        Tile qn = P.pieces[L.p[0]], qnn = P.pieces[L.p[count > 1 ? 1 : 0]];
        const int hl = tid < nvec ? tid : 0;
        double hn = st[qn.seg].h2[hl], fn = st[qn.seg].f;
        int actn = st[qn.seg].act, seg = -1, slot = -1;
        for (int k = 0; k < count; ++k) {
          const Tile q = qn;
          const double h = hn;
          const bool redo = mode == ORTH_UPD || actn == 2;
          const V f = redo ? V(1) : (V)fn;
          if (k + 1 < count) {
            qn = qnn;
            if (k + 2 < count) qnn = P.pieces[L.p[k + 2]];
            if (qn.seg != q.seg) {
              hn = st[qn.seg].h2[hl];
              fn = st[qn.seg].f;
              actn = st[qn.seg].act;
            }
          }
          V* vw = Vb + q.start + (int64_t)nvec * ld;
          if (q.seg != seg) {
            seg = q.seg;
            main_sync();
            if (tid < nvec) coef[tid] = (V)h;
            main_sync();
          }
          if constexpr (f32)
            ring_upd(ring, R, it, ok, vw, (int)(q.start & 3), q.len, nvec, coef, f);
          else
            upd_piece<V, 1, 8>(Vb + q.start, ld, nvec, vw, q.len, coef, f);
          if (redo) {  // the dots of w', which other threads of the block wrote
            const int p = L.p[k];
            if (P.slot[p] != slot) {
              slot = P.slot[p];
              for (int i = lane; i < n2; i += 32) sh.wpart[warp][i] = 0.0;
            }
            main_sync();
            dot_piece<V, LE, NB, false>(Vb + q.start, ld, nvec, vw, nullptr, q.len, P.T,
                                        sh.wpart[warp]);
            main_sync();
            if (k + 1 == count || P.slot[L.p[k + 1]] != slot) {
              store_sums(sh, part2 + (int64_t)slot * 64, n2);
              main_sync();
            }
          }
        }
      } else if constexpr (f32) {
        if (copier && lane == 0)
          for (int k = 0; k < count && ok; ++k) {
            const Tile q = P.pieces[L.p[k]];
            ok = ring_fill(Vb, ld, q.start, q.len, nvec, -1, nvec, ring, R, it);
          }
      }
    }
    if (mode == ORTH_UPD) return land();
  }
  // ---- second pass ----------------------------------------------------------
  const int nredo = mode <= ORTH_ONCE ? *(volatile int*)&ctl->nredo : 1;
  if (nredo > 0) {
    if (mode != ORTH_FIN && !meet()) return;
    for (int s = blockIdx.x; s < nseg; s += G) {
      SegState& S = st[s];
      if (mode != ORTH_FIN && S.act != 2) continue;
      __syncthreads();
      reduce_sums(sh, part2 + (int64_t)P.seg_slot[2 * s] * 64, n2, P.seg_slot[2 * s + 1], -1);
      if (warp == 0) second_column(sh, nvec, S.h2);
      __syncthreads();
      if (warp == 0) {
        if (lane < nvec) S.h2[lane] = sh.sum[lane];
        if (lane == 0) S.f = sh.f;
      }
      if (givens && mode == ORTH_STEP) {
        const V vsq = lane <= j ? gram<V>(S)[lane * 33] : V(0);
        givens_warp(S, ctl, j, m, sh.hcol, vsq);
        if (lane == 0) count_segment();
      }
    }
    if (mode != ORTH_FIN && !meet()) return;
    if (blockIdx.x == 0 && tid == 0) ctl->nredo = 0;
    for (int r = 0; r < rounds; ++r) {
      const int count = list_again(r);
      if (!work) continue;
      for (int k = 0; k < count; ++k) {
        const Tile q = P.pieces[L.p[k]];
        const SegState& S = st[q.seg];
        if (mode != ORTH_FIN && S.act != 2) continue;
        V* vw = Vb + q.start + (int64_t)nvec * ld;
        main_sync();
        if (tid < nvec) coef[tid] = (V)S.h2[tid];
        main_sync();
        upd_piece<V, 1, 8>(Vb + q.start, ld, nvec, vw, q.len, coef, (V)S.f);
      }
    }
  }
  if (blockIdx.x == 0 && tid == 0 && bars > 0) ctl->bar_base = base + bars * G;
  if (!ok && lane == 0) orth_give_up(st, ctl, nseg, cond);  // a wait ran out
  land();
}

template <typename V>
void launch_orth(V* Vb, int64_t ld, const OrthPlan& P, SegState* st, KCtl* ctl,
                 cudaGraphConditionalHandle cond, int mode, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P.blocks);
  cfg.blockDim = dim3(P.share > 0 ? kOneThreads : kManyThreads);
  cfg.dynamicSmemBytes = P.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = P.blocks > 1 ? 1 : 0;
  if (P.share == 0) {
    cudaLaunchKernelEx(&cfg, k_orth_many<V>, Vb, ld, P, st, ctl, cond, mode);
  } else if (P.LU == 1) {
    cudaLaunchKernelEx(&cfg, k_orth_one<V, 1>, Vb, ld, P, st, ctl, cond, mode);
  } else if constexpr (sizeof(V) == 4) {
    cudaLaunchKernelEx(&cfg, P.LU == 2 ? k_orth_one<V, 2> : k_orth_one<V, 4>, Vb, ld, P, st, ctl,
                       cond, mode);
  }
  count_launches(1);
}

}  // namespace

template <typename V>
int orth_blocks(bool many, int64_t* smem) {
  int dev = 0, sms = 0, per = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto fits = [&](auto k, int threads) {
    int q = 0;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k, threads, (size_t)*smem);
    per = q < per ? q : per;
  };
  if (many) {
    *smem = sizeof(V) == 4 ? (int64_t)kRingBytes : 0;
    fits(k_orth_many<V>, kManyThreads);
  } else {
    *smem = 0;
    fits(k_orth_one<V, 1>, kOneThreads);
    if constexpr (sizeof(V) == 4) {
      fits(k_orth_one<V, 2>, kOneThreads);
      fits(k_orth_one<V, 4>, kOneThreads);
    }
  }
  cudaGetLastError();
  return per * sms;
}
template int orth_blocks<double>(bool, int64_t*);
template int orth_blocks<float>(bool, int64_t*);

template <typename V>
void launch_seg_orth(V* Vb, int64_t ld, const OrthPlan& P, SegState* st, KCtl* ctl,
                     cudaGraphConditionalHandle cond, cudaStream_t s) {
  launch_orth(Vb, ld, P, st, ctl, cond, ORTH_STEP, s);
}
template void launch_seg_orth<double>(double*, int64_t, const OrthPlan&, SegState*, KCtl*,
                                      cudaGraphConditionalHandle, cudaStream_t);
template void launch_seg_orth<float>(float*, int64_t, const OrthPlan&, SegState*, KCtl*,
                                     cudaGraphConditionalHandle, cudaStream_t);

template <typename V>
void launch_seg_orth_pass(V* Vb, int64_t ld, const OrthPlan& P, SegState* st, KCtl* ctl, int pass,
                          cudaStream_t s) {
  constexpr int kMode[] = {ORTH_DOT, ORTH_UPD, ORTH_FIN, ORTH_ONCE};
  const int mode = pass < 0 ? ORTH_FULL : kMode[pass];
  launch_orth(Vb, ld, P, st, ctl, 0, mode, s);
}
template void launch_seg_orth_pass<double>(double*, int64_t, const OrthPlan&, SegState*, KCtl*,
                                           int, cudaStream_t);
template void launch_seg_orth_pass<float>(float*, int64_t, const OrthPlan&, SegState*, KCtl*, int,
                                          cudaStream_t);

}  // namespace fs
