// Drives the orthogonalisation kernels alone, on vectors, Gram matrices and
// work-lists that a test chooses (fs_orth.cu is compiled into this file).
#include "fs_orth.cu"

#include <algorithm>
#include <cstring>
#include <vector>

namespace fs {
void count_launches(int64_t) {}
}  // namespace fs

namespace {

using fs::KCtl;
using fs::OrthPlan;
using fs::SegState;
using fs::Tile;

struct Case {
  int32_t many, nseg, j, T, LU, blocks, piece, absent;
  int64_t n, share;
  uint64_t wait_ns;
};

struct Pool {
  std::vector<void*> p;
  template <typename T>
  T* up(const std::vector<T>& h) {
    T* d = nullptr;
    if (cudaMalloc((void**)&d, sizeof(T) * std::max<size_t>(1, h.size())) != cudaSuccess)
      return nullptr;
    p.push_back(d);
    cudaMemcpy(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice);
    return d;
  }
  ~Pool() {
    for (void* q : p) cudaFree(q);
  }
};

// The work-list of a batch, or of one long segment: pieces of one segment
// each, dealt to the blocks in turn; a slot of partial sums per block and
// segment, and per round of a block's list.
void plan_pieces(const Case& c, const int64_t* seg0, Pool& pool, OrthPlan& o) {
  std::vector<Tile> pieces;
  for (int s = 0; s < c.nseg; ++s)
    for (int64_t at = seg0[s]; at < seg0[s + 1]; at += c.piece) {
      Tile t{};
      t.start = at;
      t.len = (int32_t)std::min<int64_t>(c.piece, seg0[s + 1] - at);
      t.seg = s;
      pieces.push_back(t);
    }
  o.npiece = (int)pieces.size();
  o.blocks = std::min(o.blocks, o.npiece);
  std::vector<int32_t> slot(o.npiece), ss(2 * c.nseg, 0);
  for (int p = 0; p < o.npiece;) {
    const int seg = pieces[p].seg, round = p / o.blocks / fs::kOrthList;
    int e = p;
    while (e < o.npiece && pieces[e].seg == seg && e / o.blocks / fs::kOrthList == round) {
      slot[e] = o.nslot + (e - p) % o.blocks;
      ++e;
    }
    const int used = std::min(o.blocks, e - p);
    if (ss[2 * seg + 1] == 0) ss[2 * seg] = o.nslot;
    ss[2 * seg + 1] += used;
    o.nslot += used;
    p = e;
  }
  o.pieces = pool.up(pieces);
  o.slot = pool.up(slot);
  o.seg_slot = pool.up(ss);
}

template <typename V>
int plan(const Case& c, const int64_t* seg0, Pool& pool, OrthPlan& o) {
  const int cap = fs::orth_blocks<V>(c.many != 0, &o.smem);
  o.n = c.n;
  o.T = c.T;
  o.LU = c.LU;
  o.blocks = c.blocks;
  if (cap < c.blocks) return -1;
  if (c.many) {
    plan_pieces(c, seg0, pool, o);
  } else {
    o.share = c.share;
    if ((c.n + c.share - 1) / c.share != c.blocks) return -2;
  }
  o.partial = pool.up(std::vector<double>(128 * (size_t)std::max(o.nslot, o.blocks), NAN));
  return 0;
}

// The Gram correction of a segment as the kernels of type V hold it.
template <typename V>
auto* gram(SegState& S) {
  return fs::gram<V>(S);
}

std::vector<SegState> segments(const Case& c, int done) {
  std::vector<SegState> st(c.nseg);
  for (SegState& s : st) {
    memset((void*)&s, 0, sizeof(s));
    for (int i = 0; i < fs::kMaxRestart; ++i) s.cs[i] = 1.0;  // rotations of no effect
    s.g[c.j] = 1.0;
    s.done = done;
  }
  return st;
}

KCtl control(const Case& c, int done) {
  KCtl k{};
  k.m = fs::kMaxRestart;
  k.nseg = c.nseg;
  k.j = c.j;
  k.ndone = done ? c.nseg : 0;
  k.all_done = done;
  k.wait_ns = c.wait_ns;
  // arrivals that never come: every barrier of the launch waits for more
  // blocks than there are
  k.bar_base = c.absent;
  return k;
}

// One Arnoldi step's orthogonalisation of V[j + 1] against V[0..j] (rows of
// length n).  E: per segment the 32 x 32 Gram correction, in and out.
// h: per segment 33 entries, its Hessenberg column before the new rotation.
// state: the segments' records, used as they are when resume; rot: per
// segment the cosine and sine of the rotation before this step's.
template <typename V>
int step(const Case& c, const int64_t* seg0, const double* Vin, double* E, double* w, double* h,
         int32_t* seg_out, int32_t* ctl_out, void* state, int resume, double* rot) {
  Pool pool;
  OrthPlan o;
  if (int rc = plan<V>(c, seg0, pool, o)) return rc;
  const int64_t ld = (c.n + 3) / 4 * 4;
  const int rows = c.j + 2;
  std::vector<V> hv(rows * ld, (V)NAN);  // the padding is never used
  for (int r = 0; r < rows; ++r)
    for (int64_t i = 0; i < c.n; ++i) hv[r * ld + i] = (V)Vin[r * c.n + i];
  V* dV = pool.up(hv);
  std::vector<SegState> st = segments(c, 0);
  if (resume) memcpy((void*)st.data(), state, sizeof(SegState) * c.nseg);
  for (int s = 0; s < c.nseg; ++s)
    for (int i = 0; i < 1024 && !resume; ++i) gram<V>(st[s])[i] = E[1024 * s + i];
  SegState* dst = pool.up(st);
  KCtl k = control(c, 0);
  KCtl* dk = pool.up(std::vector<KCtl>{k});
  fs::launch_seg_orth<V>(dV, ld, o, dst, dk, 0, 0);
  if (cudaDeviceSynchronize() != cudaSuccess) return -3;
  cudaMemcpy(hv.data(), dV, sizeof(V) * hv.size(), cudaMemcpyDeviceToHost);
  cudaMemcpy(st.data(), dst, sizeof(SegState) * c.nseg, cudaMemcpyDeviceToHost);
  cudaMemcpy(&k, dk, sizeof(k), cudaMemcpyDeviceToHost);
  memcpy(state, st.data(), sizeof(SegState) * c.nseg);
  for (int64_t i = 0; i < c.n; ++i) w[i] = (double)hv[(rows - 1) * ld + i];
  for (int s = 0; s < c.nseg; ++s) {
    const SegState& S = st[s];
    for (int i = 0; i < 1024; ++i) E[1024 * s + i] = (double)gram<V>(st[s])[i];
    for (int i = 0; i < c.j; ++i) h[33 * s + i] = S.H[i * k.m + c.j];
    const double den = S.H[c.j * k.m + c.j];
    h[33 * s + c.j] = S.cs[c.j] * den;
    h[33 * s + c.j + 1] = S.sn[c.j] * den;
    rot[2 * s] = c.j > 0 ? S.cs[c.j - 1] : 1.0;
    rot[2 * s + 1] = c.j > 0 ? S.sn[c.j - 1] : 0.0;
    const int32_t out[4] = {S.bad, S.done, S.act, S.k};
    std::copy(out, out + 4, seg_out + 4 * s);
  }
  const int32_t out[4] = {k.j, k.all_done, k.nredo, (int32_t)k.bar};
  std::copy(out, out + 4, ctl_out);
  return 0;
}

// A pass counter that ends the loop after max_pass passes whatever the kernel
// before it did.
__global__ void k_fuse(int* pass, int max_pass, cudaGraphConditionalHandle cond) {
  if (++*pass >= max_pass) cudaGraphSetConditional(cond, 0);
}

// The Arnoldi loop node entered with its condition set and every segment
// done, as a block that re-armed the condition behind a wait that ran out
// leaves it: the passes it takes.
template <typename V>
int loop(const Case& c, const int64_t* seg0, int max_pass, int* passes) {
  Pool pool;
  OrthPlan o;
  if (int rc = plan<V>(c, seg0, pool, o)) return rc;
  const int64_t ld = (c.n + 3) / 4 * 4;
  V* dV = pool.up(std::vector<V>((c.j + 2) * ld, V(0)));
  SegState* dst = pool.up(segments(c, 1));
  KCtl* dk = pool.up(std::vector<KCtl>{control(c, 1)});
  int* dp = pool.up(std::vector<int>{0});
  cudaStream_t s;
  cudaStreamCreate(&s);
  cudaGraph_t g, body, got;
  cudaGraphCreate(&g, 0);
  cudaGraphConditionalHandle cond;
  cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault);
  cudaGraphNodeParams np = {};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = cond;
  np.conditional.type = cudaGraphCondTypeWhile;
  np.conditional.size = 1;
  cudaGraphNode_t node;
  cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np);
  body = np.conditional.phGraph_out[0];
  cudaStreamBeginCaptureToGraph(s, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
  fs::launch_seg_orth<V>(dV, ld, o, dst, dk, cond, s);
  k_fuse<<<1, 1, 0, s>>>(dp, max_pass, cond);
  cudaStreamEndCapture(s, &got);
  cudaGraphExec_t x = nullptr;
  int rc = cudaGraphInstantiate(&x, g, 0) == cudaSuccess ? 0 : -4;
  if (rc == 0) {
    cudaGraphLaunch(x, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) rc = -3;
    cudaMemcpy(passes, dp, sizeof(int), cudaMemcpyDeviceToHost);
    cudaGraphExecDestroy(x);
  }
  cudaGraphDestroy(g);
  cudaStreamDestroy(s);
  return rc;
}

}  // namespace

extern "C" {
int orth_state_size() { return (int)sizeof(SegState); }
int orth_step(int f32, const void* c, const int64_t* seg0, const double* V, double* E, double* w,
              double* h, int32_t* seg_out, int32_t* ctl_out, void* state, int resume,
              double* rot) {
  return f32 ? step<float>(*(const Case*)c, seg0, V, E, w, h, seg_out, ctl_out, state, resume, rot)
             : step<double>(*(const Case*)c, seg0, V, E, w, h, seg_out, ctl_out, state, resume, rot);
}
int orth_loop(int f32, const void* c, const int64_t* seg0, int max_pass, int* passes) {
  return f32 ? loop<float>(*(const Case*)c, seg0, max_pass, passes)
             : loop<double>(*(const Case*)c, seg0, max_pass, passes);
}
}
