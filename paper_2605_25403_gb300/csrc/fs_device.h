// Launchers of the sm_103a kernels (defined in fs_assembly.cu and
// fs_linalg.cu) and the plain views they take.  Host code only sees these
// declarations; every pointer in a view is a device pointer.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

#include "fs_internal.h"

namespace fs {

// Counts kernel launches issued from the host (ignored while a stream is
// being captured into a graph; graph replays add their node count).
void count_launches(int64_t n);

// Programmatic dependent launch.  The solver's kernels run as chains of
// short dependent passes (a V-cycle's levels, the Gram-Schmidt passes), so
// the gap between one kernel's last block and the next kernel's first is a
// large part of a step.  A kernel launched by launch_k with the overlap mode
// on may be scheduled while its predecessor in the stream drains; its first
// statement is pdl_wait() (griddepcontrol.wait), which returns once every
// prerequisite grid has completed and its memory operations are visible, so
// no global access of the kernel can overlap the predecessor.  Without the
// attribute griddepcontrol.wait returns at once and the launch is an
// ordinary serialised one.  The mode is per calling thread, taken from the
// problem's schedule by the API entry points.
bool launch_overlap();

// Limit of a wait inside a kernel: one second (fs_set_wait_limit changes a
// problem's).  A kernel whose wait runs out marks its result and returns, and
// the call reports FS_ERR_TIMEOUT.
constexpr uint64_t kWaitNs = 1000000000ull;

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// All blocks of a cooperative launch (which guarantees that they are resident
// together) arrive before any leaves; false in every thread when the wait has
// not ended after `limit` ns.  target counts the arrivals since the counter's
// reset, modulo 2^32; ok: a word of shared memory.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned target, uint64_t limit,
                                             int* ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    *ok = 1;
    if (gridDim.x > 1) {
      __threadfence();
      atomicAdd(bar, 1u);
      const uint64_t t0 = now_ns();
      unsigned v;
      while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if ((int)(v - target) >= 0) break;
        if (now_ns() - t0 >= limit) {
          *ok = 0;
          break;
        }
      }
    }
  }
  __syncthreads();
  return *ok != 0;
}
#endif

template <typename... KArgs, typename... Args>
inline void launch_k(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                     Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = launch_overlap() ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

// Element-level reference integrals in constant memory (per dimension).
void upload_ref_tensors(const RefTensors& R2, const RefTensors& R3);

template <typename T>
struct DCsr {
  int32_t nrow = 0;
  // threads that share a row in the transfer kernels (1, 4 or 32, from the
  // mean row length: one thread per row for the 1-3 entries of a
  // prolongation row, a warp for the ~50 of a restriction row onto a grid
  // coarsened by 4)
  int32_t lanes = 4;
  const int32_t* rp = nullptr;
  const int32_t* ci = nullptr;
  const T* v = nullptr;
};

// Sliced ELLPACK with slices of 32 rows (one thread per row): the entries of
// row 32 s + t sit at off[s] + 32 u + t for the slot u < (off[s+1] - off[s]) / 32,
// so a warp's loads of one slot are contiguous.  Slots a row does not use hold
// the coefficient -0.0 and a valid column; the row's own entries are never
// -0.0, so that a product can leave the others out where 0 x Inf would matter
// (a run's padding columns belong to other rows' stencils).
//
// Columns.  Consecutive rows of a structured mesh have the same stencil
// shifted by one, so a slice's slots can be laid out by column offset: in a
// slice with a split > 0 the column of slot u is runs[off / 32 + u].x + t for
// t < split (the rows of one grid line) and .y + t from there on (those of the
// next line), 8 bytes per slot instead of 128 and already in L1 for the next
// slot.  split = 0 (short grid lines, boundary corners): the columns are read
// from ci, which always holds them.  Which slices qualify is found from the
// pattern alone.  The split travels in the top byte of the slice's offset,
// so that it costs no load of its own (a separate array of splits put one
// more load before the first gather and made the passes on small levels
// slower); layouts of one width (width > 0, the P1 levels) read no offsets
// and keep ci (runs = null).
constexpr int kSellSplit = 56;  // bit position of the split in an offset
template <typename T>
struct DSell {
  int64_t nrow = 0;
  const int64_t* off = nullptr;
  const int32_t* ci = nullptr;
  const T* v = nullptr;
  // > 0: every slice has this many slots (off[s] = 32 s width), so a
  // thread finds its slice without loading off
  int64_t width = 0;
  const int2* runs = nullptr;
};

#ifdef __CUDACC__
// One thread's view of its row: the slice's first slot and slot count, and
// where the columns come from.
template <typename T>
struct SellRow {
  int64_t first;
  int w, t, split;
  __device__ __forceinline__ SellRow(const DSell<T>& A, int64_t row) {
    const int64_t sl = row >> 5;
    t = (int)(row & 31);
    if (A.width) {
      split = 0;
      first = sl * 32 * A.width;
      w = (int)A.width;
    } else {
      constexpr int64_t kMask = ((int64_t)1 << kSellSplit) - 1;
      const int64_t a = A.off[sl], b = A.off[sl + 1];
      split = (int)(a >> kSellSplit);
      first = a & kMask;
      w = (int)(((b & kMask) - first) >> 5);
    }
  }
  // body(col, shift): the column of slot u is col(u) + shift, with shift the
  // same for every slot (a body adds it to its vector's address once).
  template <typename F>
  __device__ __forceinline__ void with_columns(const DSell<T>& A, F body) const {
    if (split > 0) {
      const int32_t* __restrict__ q =
          reinterpret_cast<const int32_t*>(A.runs + (first >> 5)) + (t < split ? 0 : 1);
      body([q](int u) { return __ldg(q + 2 * u); }, t);
    } else {
      const int32_t* __restrict__ q = A.ci + first + t;
      body([q](int u) { return __ldg(q + 32 * u); }, 0);
    }
  }
};
#endif

// A vector addressed through the device-side Arnoldi step index: base +
// (*j) stride (base itself when j is null).  The kernels of one Arnoldi step
// take their Krylov vectors this way, so that one captured step can be
// replayed by a conditional loop node while j advances on the device.
template <typename T>
struct JVec {
  T* base = nullptr;
  const int* j = nullptr;
  int64_t stride = 0;
  JVec() = default;
  JVec(T* b) : base(b) {}
  JVec(T* b, const int* jj, int64_t st) : base(b), j(jj), stride(st) {}
  JVec<T> shifted(int64_t o) const { return JVec<T>(base + o, j, stride); }
  __device__ __forceinline__ T* get() const { return j ? base + (int64_t)(*j) * stride : base; }
};

// Mesh tables and block patterns of one problem on the device.
struct DMesh {
  int dim = 0, nloc = 0, nb = 0;
  int64_t nv = 0, n2 = 0, ncell = 0;
  const int32_t* c2d = nullptr;        // ncell x nloc
  const double* p2xyz = nullptr;       // n2 x dim
  const uint8_t* dirichlet = nullptr;  // n2
  const int32_t* dlist = nullptr;      // Dirichlet node ids
  int64_t ndir = 0;
  const int32_t *rpA = nullptr, *ciA = nullptr;    // P2-P2
  const int32_t *rpB = nullptr, *ciB = nullptr;    // P1-P2
  const int32_t *rpBT = nullptr, *ciBT = nullptr;  // P2-P1
  const int32_t *rpK = nullptr, *ciK = nullptr;    // P1-P1
  const uint8_t *posA = nullptr, *posB = nullptr, *posBT = nullptr, *posK = nullptr;
  const double* nu_cell = nullptr;     // per-cell viscosity (batches) or null
  const int32_t* color_cells = nullptr;  // cells grouped by colour (Mesh)
};

// Physical description of the manufactured problem.
struct DPhys {
  int kind = 0;
  double nu = 1.0;
  const double* nu_node = nullptr;  // per-P2-node viscosity (batches) or null
  double wconst[3] = {0, 0, 0};
};

// ---- assembly (fs_assembly.cu) -------------------------------------------
// Colour-ordered element kernels (color_ptr: the host copy of
// Mesh::color_ptr, one launch per colour): the cells of a colour share no
// node, so they add into the block values with plain read-modify-writes, no
// atomics, and every value is summed in the same order on every run.
// Step-invariant blocks (always colour-ordered), accumulated into zeroed
// arrays:
// base = mass_coef M + nu K (P2-P2), Mv = M, B (P1-P2, dim values per entry),
// BT (P2-P1, dim values), Kp (P1 stiffness), mpl (lumped P1 mass).
void launch_assemble_base(const DMesh& m, const std::vector<int64_t>& color_ptr,
                          double mass_coef, double nu, double* base, double* Mv, double* B,
                          double* BT, double* Kp, double* mpl, cudaStream_t s);
// valA += N(w) with w taken from the component-blocked vector w (ldw =
// component stride) or the constant field wc when w == nullptr; rows of
// Dirichlet nodes are skipped.  deterministic: colour by colour as the
// step-invariant blocks, a thread per (cell, row); otherwise one launch over
// all cells, a thread per cell, FP64 atomics (faster; the last bits of a
// value depend on the order its contributions arrive in).
void launch_assemble_conv(const DMesh& m, const std::vector<int64_t>& color_ptr,
                          const double* w, int64_t ldw, const double* wc, double* valA,
                          bool deterministic, cudaStream_t s);
// Np += the pressure-space convection int psi_q (w . grad psi_s) (P1-P1
// pattern, slot tables posK; w component-blocked with stride ldw, or the
// constant field wc when w == nullptr); rows of the vertices with fixed set
// stay untouched.  FP64 atomics.
void launch_assemble_conv_p1(const DMesh& m, const double* w, int64_t ldw, const double* wc,
                             const uint8_t* fixed, double* Np, cudaStream_t s);
// Dirichlet rows of the scalar block become identity rows.
template <typename T>
void launch_bc_rows(const DMesh& m, T* valA, cudaStream_t s);
// F[c][j] = mass_coef * u_c[j] + f_c(x_j, t) for every P2 node.
void launch_eval_load(const DMesh& m, const DPhys& ph, double t,
                      double mass_coef, const double* u, double* F,
                      cudaStream_t s);
// b = M F (velocity rows), Dirichlet rows = u_exact(t), b_p = 0 except the
// pinned rows (p_exact at their vertex).
void launch_rhs(const DMesh& m, const DPhys& ph, double t, const double* Mv,
                const double* F, const int32_t* pinned, int npinned, double* b,
                cudaStream_t s);
// Exact state I_h u, I_h p at time t (zero_interior: 0 off Dirichlet nodes).
void launch_exact_state(const DMesh& m, const DPhys& ph, double t,
                        int zero_interior, double* x, cudaStream_t s);
// Monolithic CSR values from the block values (export for parity checks).
// Monolithic CSR values in paper order (rows and columns of fs_dof_map):
// mrp holds that CSR's row pointers and nat the paper id of each internal
// P2 node; an entry's place in its row is the rank of its paper column.
void launch_expand_monolithic(const DMesh& m, const int32_t* nat, const double* valA,
                              const double* B, const double* BT, const double* diagp,
                              const int64_t* mrp, double* out, cudaStream_t s);
// n_dof vectors between the internal and the paper order of the P2 nodes:
// to_nat = 1: out[c n2 + nat[q]] = in[c n2 + q]; to_nat = 0: the inverse;
// pressure entries are copied.
void launch_dofs_perm(const DMesh& m, const int32_t* nat, const double* in, double* out,
                      int to_nat, cudaStream_t s);

// ---- Taylor-Hood P3/P2 on triangles (fs_assembly.cu) ----------------------
// m: a DMesh holding the P3 tables (c2d = the P3 map, 10 per cell; n2 = P3
// nodes; nv = P2 pressure nodes; p2xyz = P3 node coordinates; patterns and
// slot tables of P3Tables), c2p the P2 map (6 per cell), R the reference
// integrals in device memory.  Blocks as launch_assemble_base /
// launch_assemble_conv (FP64 atomics).
void launch_p3_base(const DMesh& m, const int32_t* c2p, const RefP3* R, double mass_coef,
                    double nu, double* base, double* Mv, double* B, double* BT, double* Kp,
                    cudaStream_t s);
void launch_p3_conv(const DMesh& m, const RefP3* R, const double* w, int64_t ldw,
                    const double* wc, double* valA, cudaStream_t s);
void launch_p3_exact_state(const DMesh& m, const DPhys& ph, double t, int zero_interior,
                           const double* pxyz, double* x, cudaStream_t s);

// ---- linear algebra (fs_linalg.cu) ---------------------------------------
// Saddle-point operator in block form.
struct SegState;

// Rows of a batch whose segment (instance) has converged in the current
// restart cycle: the union kernels skip them.  slice_seg[s] is the segment
// of rows 32 s .. 32 s + 31 of a level (-1 where a slice holds rows of two
// instances: never skipped); st is the Krylov segment state (null: nothing
// is skipped, as for single problems and for timing runs).
struct SegSkip {
  const int32_t* slice_seg = nullptr;
  const SegState* st = nullptr;
};

template <typename T>
struct DOp {
  int dim = 0;
  int64_t n2 = 0, nv = 0;
  // SELL-32 blocks.  B and BT hold dim values per slot, component-major
  // within a slot: the value of component c of row 32 s + t at slot u is at
  // (off[s] + 32 u) dim + 32 c + t.
  DSell<T> A, B, BT;
  const T* diagp = nullptr;
  int group = 0;  // slots issued together per thread (0: the default)
  // batches: segments of the velocity rows (union node order) and of the
  // pressure rows, for the Arnoldi steps' products
  SegSkip skip_u, skip_p;
};

// y = K x (resid == 0) or y = b - K x (resid == 1); vectors of type V.
// exact (FP64): the padding slots take no part, not even as 0 x Inf.
// seg: skip the rows of converged segments (the Arnoldi step's product;
// residuals and timing runs take every row).
template <typename T, typename V>
void launch_spmv_full(const DOp<T>& op, JVec<const V> x, const V* b, JVec<V> y,
                      int resid, const int* skip, cudaStream_t s, bool seg = false,
                      bool exact = false);

// Scalar CSR values (row pointers rp, columns ci) into the SELL-32 layout L
// (its offsets and columns): out64 (and out32 when not null) receive the
// matrix, -0.0 in the slots a row does not use.
void launch_csr_to_sell(const DSell<double>& L, const int32_t* rp, const int32_t* ci,
                        const double* in, double* out64, float* out32, cudaStream_t s);

// Multigrid level on the device.
template <typename T>
struct DLevel {
  DSell<T> A;           // level operator
  DCsr<T> P, R;         // P: prolongation from level+1, R = P^T
  SegSkip skip;         // rows of this level by segment
  const T* dinv = nullptr;
  double inv_theta = 0, a1 = 0, b1 = 0, a2 = 0, b2 = 0;  // Chebyshev(3)
  double lmax = 0;  // estimate of the largest eigenvalue of D^-1 A (host set-up)
};
template <typename T>
struct DHier {
  int nlev = 0;
  int ncp = 1;  // components per row in the level vectors (1, 2 or 4)
  DLevel<T> lev[16];
  // coarsest level: block-diagonal dense inverses (one block per instance)
  const T* cinv = nullptr;           // concatenated row-major blocks
  const int32_t* row_blk = nullptr;  // coarsest row -> block
  const int64_t* blk_row = nullptr;  // block -> first row
  const int64_t* blk_n = nullptr;    // block -> size
  const int64_t* blk_dense = nullptr;  // block -> offset in cinv
  int64_t ncoarse = 0;
  int64_t dense_nb0 = 0;  // ncoarse when the coarsest level is one block, else 0
  // per level (all rows x ncp, row-interleaved components): right-hand
  // side b, and ping-pong pairs of the gather vector G (x + d, the point the
  // next residual is taken at) and the Chebyshev direction D
  T* b[16] = {};
  T* G0[16] = {};
  T* G1[16] = {};
  T* D0[16] = {};
  T* D1[16] = {};
  // level-0 block order vs the caller's vector order (batches): perm[r] is
  // the caller's row of block row r, iperm its inverse; null when equal
  const int32_t* perm = nullptr;
  const int32_t* iperm = nullptr;
  // slots issued together per thread in the smoothing passes (4 or 6; 0: by
  // precision and level)
  int group = 0;
  // Chebyshev degree of the pre- and post-smoothing below the finest level
  // and on the finest level (3 or 2 each)
  int coarse_deg = 2;
  int fine_deg = 3;
  // first level run by the fused cluster kernel (-1: none), its cluster size
  int tail = -1;
  int tail_cluster = 8;
  double fine_index_bytes = 0;  // offsets and columns a pass over level 0 reads
  // a copy of this struct in device memory (read by the coarse kernels)
  const DHier<T>* dev = nullptr;
};

// The hierarchy with segment skipping off (timing and profiling runs, whose
// segment states are those of the last solve).
template <typename T>
inline DHier<T> without_skip(const DHier<T>& H) {
  DHier<T> C = H;
  for (int l = 0; l < 16; ++l) C.lev[l].skip.st = nullptr;
  return C;
}

// Gauss-Jordan inversion with partial pivoting of a dense n x n FP64
// matrix, held row-major as the augmented n x 2n array W = [A | I]; after
// the n pivot steps the right half holds A^-1 (the left half is not kept
// up to date).  piv, pval: device scratch for the pivot row and value; bad:
// device flag set when a pivot column is zero.  Set-up only.
void launch_gj_step(double* W, int64_t n, int64_t c, int64_t* piv, double* pval, int* bad,
                    cudaStream_t s);
// out (n x n, row-major) = the right half of W, converted to T.
template <typename T>
void launch_gj_extract(const double* W, int64_t n, T* out, cudaStream_t s);

// Cluster size (16 or 8 blocks) of the fused kernel for this arithmetic and
// row width.
template <typename T>
int mg_tail_cluster(int ncp);

// One fused Chebyshev step (mode STEP) on level 0 of H with its own work
// vectors, for kernel timing.
template <typename T>
void launch_cheb_step(const DHier<T>& H, int nc, cudaStream_t s);

// scratch[0] = sum_i (a_i - b_i)^2, scratch[1] = sum_i a_i^2 over i < n, in
// a fixed summation order; scratch holds diff_norms_scratch() doubles.
int diff_norms_scratch();
void launch_diff_norms(const double* a, const double* b, int64_t n, double* scratch,
                       cudaStream_t s);

// Reads `bytes` (a multiple of 16) of buf so that the L2 holds clean lines
// of it and nothing of the data timed next (kernel timing with a cold L2).
void launch_l2_flush(const void* buf, int64_t bytes, int* sink, cudaStream_t s);

// Polynomial extrapolation in time of the state x (x^n) through it and its
// nprev <= kExtrapMax previous values prev[j] = x^(n-1-j) to the next time
// level: x <- sum_j (-1)^j C(nprev+1, j+1) x^(n-j) over j = 0..nprev (x
// itself for nprev = 0); the old x goes to dst, which may be prev[nprev-1]
// (each entry is read before it is written).  n entries each.
void launch_extrapolate(double* x, const double* const* prev, int nprev, double* dst, int64_t n,
                        cudaStream_t s);

// Conversion out = (B)(in * scale) (scale = *scale or 1/*scale when inv).
template <typename A, typename B>
void launch_convert(const A* in, B* out, int64_t n, const double* scale,
                    int inv, cudaStream_t s);

// The convection part of the pressure convection-diffusion operator, for
// the Schur-complement approximation: the P1-P1 matrix Np (CSR rows of the
// pressure vertices) and the inverse lumped pressure mass.  v == nullptr:
// not used.
template <typename T>
struct PcdView {
  const int32_t* rp = nullptr;
  const int32_t* ci = nullptr;
  const T* v = nullptr;
  const T* invm = nullptr;
};

// z = P^-1 r, the block preconditioner.  mpl_inv_nu: nu over the lumped
// pressure mass per vertex, negative on the pinned vertices (their rows pass
// r_p through).  With pcd.v set, the Schur part is
// M_p^-1 (M_p / dt + nu K_p + N_p) K_p^-1 (pressure convection-diffusion)
// instead of nu M_p^-1 + dt^-1 K_p^-1 (Cahouet-Chabard).
template <typename T>
void launch_precond(const DOp<T>& op, const DHier<T>& HA, const DHier<T>& HK,
                    const T* mpl_inv_nu, double inv_dt, JVec<const T> r, JVec<T> z,
                    T* work_p, T* work_u,
                    const int* skip, cudaStream_t s, const PcdView<T>& pcd = PcdView<T>());

// ---- the block preconditioner as one persistent kernel (fs_linalg.cu) ----
// The passes of launch_precond (pressure load, the pressure V-cycle, the
// Cahouet-Chabard combination, the B^T coupling, the velocity V-cycle) become
// phases of a work-list of items (phase, instance, row range).  One
// cooperative launch (every block resident) walks it: block b takes items
// b, b + grid, ... in list order; an item of phase p of instance i starts
// once every item of phase p - 1 of instance i has finished (a counter per
// (phase, instance), incremented after each item with release semantics,
// polled with acquire loads by the block's first thread).  Instances are
// independent (every operator of a batch is block-diagonal), so no phase
// waits for the whole batch.  Items of instances that converged in the
// running cycle are skipped.  The list is ordered by phase, so every item's
// predecessors come before it and, all blocks being resident, every wait
// ends; each wait still gives up after one second (the segment is then
// marked with bad = 2 and the solve reports FS_ERR_TIMEOUT).  The last
// block to leave zeroes the counters for the next launch.
struct FlowItem {
  int32_t phase, seg, row0, row1;
};
struct FlowHost {
  std::vector<unsigned char> phases;  // nphase phase records (fs_linalg.cu)
  std::vector<FlowItem> items;
  std::vector<int32_t> need;          // items per (phase, instance): nphase x nseg
  int nphase = 0;
};
struct FlowDev {
  const void* phases = nullptr;
  const FlowItem* items = nullptr;
  int64_t nitems = 0;
  unsigned* cnt = nullptr;             // nphase x nseg, zero between launches
  const int32_t* need = nullptr;
  unsigned* ticket = nullptr;          // exit ticket, zero between launches
  int nphase = 0, nseg = 0, nblocks = 0;
};
// Resident blocks of the persistent kernel for this arithmetic and velocity
// row width (ncp 2 or 4): blocks per SM x SMs of the current device.
template <typename T>
int flow_blocks(int ncp);
// The work-list of one application.  offA / offK: per level of HA / HK the
// first row of each instance (nseg + 1 entries, block order); prow: the
// first caller pressure row of each instance (nseg + 1).  Items are
// sized so that a phase over all instances has at least `nblocks` of them
// when it has enough rows.
template <typename T>
void build_flow(const DHier<T>& HA, const DHier<T>& HK,
                const std::vector<std::vector<int64_t>>& offA,
                const std::vector<std::vector<int64_t>>& offK, const std::vector<int64_t>& prow,
                int nblocks, FlowHost& out);
// One application through the persistent kernel (same arguments as
// launch_precond, plus the plan; st: skip instances with done set, or null;
// flag: segment states that receive bad = 2 on a timed-out wait, or null).
template <typename T>
void launch_precond_flow(const FlowDev& f, const DOp<T>& op, const DHier<T>& HA,
                         const T* mpl_inv_nu, double inv_dt, JVec<const T> r, JVec<T> z,
                         T* work_p,
                         const SegState* st, SegState* flag, const int* skip, cudaStream_t s);

// ---- incremental pressure correction (fs_ipcs.cu) -----------------------
// Right-hand sides of the three stages (x = [u^n | p^n], b = the assembled
// load with the Dirichlet and pinned values of t^{n+1}); see fs_ipcs.cu.
void launch_ipcs_rhs1(const DMesh& m, const double* valA, const double* base, const double* BT,
                      const double* b, const double* x, double* r, cudaStream_t s);
void launch_ipcs_rhs2(const DMesh& m, const double* B, const double* ustar, double inv_dt,
                      const uint8_t* fixed, const double* b, const double* x, double* r,
                      cudaStream_t s);
void launch_ipcs_rhs3(const DMesh& m, const double* Mv, const double* BT, const double* b,
                      const double* ustar, const double* dp, double dt, double* r,
                      cudaStream_t s);
// y = A x for which = 0 (scalar P2 block `vals` on every component,
// identity at Dirichlet nodes) or 1 (P1 Laplacian `vals`, identity at the
// fixed vertices); part (may be null) receives per-block partials of x . y;
// returns the number of blocks.
int launch_ipcs_apply(const DMesh& m, int which, const double* vals, const uint8_t* fixed,
                      const double* x, double* y, double* part, cudaStream_t s);
void launch_ipcs_dinv(const DMesh& m, int which, const double* vals, const uint8_t* fixed,
                      double* dinv, cudaStream_t s);
void launch_ipcs_fix(const DMesh& m, int which, const uint8_t* fixed, const double* rhs,
                     double* x, cudaStream_t s);
void launch_ipcs_add(int64_t n, const double* x, double* y, cudaStream_t s);
// doubles of block-partial scratch the CG kernels need on this mesh
int ipcs_part_size(const DMesh& m);
// A whole Jacobi-preconditioned CG solve of the stage `which` (0: DIM
// components, 1: pressure) as one cooperative launch: op the operator, x the
// guess with its fixed unknowns in place, dinv the inverse diagonal, part
// ipcs_part_size doubles; ctl receives the iterations, the squared norms of
// the true residual and of rhs, and bad = 1 when a wait ran out.
constexpr int kCgMaxBlocks = 256;
struct CgCtl {
  unsigned bar;
  int iters, bad, pad;
  double rr, bb;
};
struct CgOp {
  int64_t n = 0;                   // rows
  const uint8_t* fixed = nullptr;  // identity rows
  DSell<double> sell;              // used when its values are set, else CSR:
  const int32_t *rp = nullptr, *ci = nullptr;
  const double* v = nullptr;
};
void launch_cg_solve(const DMesh& m, int which, const CgOp& op, const double* rhs, double* x,
                     const double* dinv, double* r, double* z, double* p, double* p2,
                     double* q, double* part, CgCtl* ctl, double rtol, int max_iter,
                     uint64_t wait_ns, cudaStream_t s);
// The V-cycle-preconditioned pressure stage, a kernel per step; sc (4 doubles
// on the device): rz, alpha, beta, rr.
void launch_cg_init(int64_t n, const double* rhs, const double* y, const double* dinv, double* r,
                    double* z, double* p, double* part, double* sc, cudaStream_t s);
void launch_cg_alpha(const double* part, int nb, double* sc, cudaStream_t s);
void launch_cg_dir(int64_t n, const double* sc, const double* z, double* p, cudaStream_t s);
// Flexible CG (preconditioner applied by the caller between the two):
// t = r, x += alpha p, r -= alpha q (rr into sc[3]); then with z = M(r),
// zeroed on the fixed rows, the dots r.z, t.z give beta (Polak-Ribiere) and
// the new rz; first = 1 starts the iteration (p = z, rz = r.z).
void launch_cg_update_flex(int64_t n, double* sc, const double* p, const double* q, double* x,
                           double* r, double* t, double* part, cudaStream_t s);
void launch_cg_dots_flex(int64_t n, const uint8_t* fixed, const double* r, const double* t,
                         double* z, double* p, int first, double* part, double* sc,
                         cudaStream_t s);

// z = one V-cycle of the single-component hierarchy H on r (n level-0 rows
// in the caller's order): the pressure Laplacian part of the block
// preconditioner, reused to precondition the IPCS pressure increment.
template <typename T>
void launch_vcycle_scalar(const DHier<T>& H, const T* r, T* z, int64_t n, cudaStream_t s);

// ---- segmented Krylov (fs_krylov.cu) -------------------------------------
constexpr int kTileLen = 2048;  // vector entries per reduction tile

// A contiguous range [start, start + len) of one segment's entries.
struct Tile {
  int64_t start;
  int32_t len;
  int32_t seg;
};
struct TileList {
  const Tile* tiles = nullptr;
  int ntiles = 0;
};

// Per-segment state of the restart cycle.  The first 64 bytes are the
// status block the host reads back after every part of a solve.
struct SegState {
  double beta;      // ||r0|| of the cycle
  double resid;     // Arnoldi residual estimate
  double bnorm;     // ||b|| (FP64 right-hand side of the segment)
  double rnorm;     // FP64 residual norm (refinement)
  double tol_abs;   // Arnoldi target of the cycle
  int done;         // converged / retired / broken: kernels skip the segment
  int k;            // Arnoldi steps taken in this cycle
  int bad;          // NaN/Inf seen
  int retired;      // set by the host: the segment no longer iterates
  int first_tile, ntiles;
  double rtol;      // set by the host: target of the next cycle, relative to
                    // beta or to bnorm (device data, so captured graphs stay
                    // valid when it changes)
  unsigned counter[8];
  double H[(kMaxRestart + 1) * kMaxRestart];
  double cs[kMaxRestart], sn[kMaxRestart], g[kMaxRestart + 1];
  double h2[kMaxRestart + 1];  // coefficients of the running update
  double f;                    // and 1 / ||w|| (orthogonalisation by pieces),
  int act;                     // 0: not active, 1: active, 2: second pass needed
  // V^T V - I of the cycle's basis (symmetric), 32 x 32 in the vectors' type
  double E[32 * 32];
};
#ifdef __CUDACC__
__device__ __forceinline__ bool seg_skipped(const SegSkip& k, int64_t row) {
  if (!k.st) return false;
  const int32_t g = k.slice_seg[row >> 5];
  return g >= 0 && k.st[g].done;
}
#endif

struct KCtl {
  int m;         // restart length
  int nseg;      // number of segments
  int ndone;     // segments done in this cycle
  int all_done;  // every segment done: the spanning kernels skip
  int j;         // Arnoldi step of the cycle (reset by the cycle init,
                 // advanced by the Givens step)
  int nfin;      // segments whose Givens step of this column is taken
  int nredo;     // segments whose orthogonalisation needs a second pass
  unsigned bar, bar_base;  // grid barrier of the orthogonalisation kernel:
                           // arrivals, and their count before the launch
  uint64_t wait_ns;        // limit of each of that kernel's waits
};

template <typename V>
void launch_seg_norm(const V* x, const TileList& tl, SegState* st, double* partial,
                     int field, cudaStream_t s);
// cond: the handle of a conditional loop node replaying the Arnoldi step
// (0 when the steps are launched one by one); the cycle init sets it to
// "not every segment done", the orthogonalisation to "not done and j < m".
void launch_seg_cycle_init(SegState* st, KCtl* ctl, int relative_to_beta,
                           cudaGraphConditionalHandle cond, cudaStream_t s);
template <typename V>
void launch_seg_scale(JVec<V> x, const TileList& tl, const SegState* st, cudaStream_t s);
// How the entries of the n_dof vectors are dealt to the blocks of the
// orthogonalisation kernels (fs_orth.cu).  share > 0: one segment, block b
// holds the entries from b share on.  share = 0: pieces of one segment each,
// dealt to the blocks in turn, a slot of partial sums per piece.
struct OrthPlan {
  int blocks = 0;
  int64_t n = 0;        // entries of a vector
  int T = 512, LU = 4;  // dot pass: threads per group; update: entries per thread
  int64_t share = 0;
  int64_t smem = 0;     // dynamic shared memory, bytes
  int npiece = 0, nslot = 0;
  const Tile* pieces = nullptr;
  const int32_t* slot = nullptr;      // per piece: the slot of its block and segment
  const int32_t* seg_slot = nullptr;  // per segment: first slot, count
  double* partial = nullptr;          // 128 per block (share > 0) or per slot
};
constexpr int kOrthPiece = 2048;  // entries of a piece at most
constexpr int kOrthList = 1024;   // pieces a block lists at a time
// Blocks of the orthogonalisation kernel (the one for pieces when many) that
// are resident together, and the dynamic shared memory each may use.
template <typename V>
int orth_blocks(bool many, int64_t* smem);
// Orthogonalises w = V[j + 1] (j = ctl->j; vectors ld apart, a multiple of
// 4) against V[0..j] and normalises it, takes the Givens step of column j of
// every active segment and advances the step index (setting cond when not
// 0).  One cooperative launch.
template <typename V>
void launch_seg_orth(V* Vb, int64_t ld, const OrthPlan& P, SegState* st, KCtl* ctl,
                     cudaGraphConditionalHandle cond, cudaStream_t s);
// For kernel timing, without the Givens step: the orthogonalisation with its
// second pass always taken (pass < 0) or never (3), or its dot pass (0), its
// update pass with the re-dots (1) or its second pass (2) alone.
template <typename V>
void launch_seg_orth_pass(V* Vb, int64_t ld, const OrthPlan& P, SegState* st, KCtl* ctl, int pass,
                          cudaStream_t s);
template <typename V, typename X>
void launch_seg_update_x(const SegState* st, const KCtl* ctl, const V* Z, int64_t n,
                         const TileList& tl, X* x, cudaStream_t s);
template <typename A, typename B>
void launch_seg_normalise(const A* in, B* out, const TileList& tl, const SegState* st,
                          cudaStream_t s);
template <typename V, typename X>
void launch_seg_axpy(X* x, const V* d, const TileList& tl, const SegState* st,
                     cudaStream_t s);

}  // namespace fs
