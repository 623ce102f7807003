// Drives the one-launch Jacobi-CG solve alone (fs_ipcs.cu is compiled into this
// file), with blocks that never come when absent > 0.
#include "fs_ipcs.cu"

#include <vector>

namespace fs {
void count_launches(int64_t) {}
bool launch_overlap() { return false; }
}  // namespace fs

namespace {
struct Pool {
  std::vector<void*> p;
  template <typename T>
  T* up(const T* h, size_t n) {
    T* d = nullptr;
    if (cudaMalloc((void**)&d, sizeof(T) * n) != cudaSuccess) return nullptr;
    p.push_back(d);
    cudaMemcpy(d, h, sizeof(T) * n, cudaMemcpyHostToDevice);
    return d;
  }
  ~Pool() {
    for (void* q : p) cudaFree(q);
  }
};
}  // namespace

// n rows in CSR, one component; out: iterations, bad.
extern "C" int cg_solve(int64_t n, const int32_t* rp, const int32_t* ci, const double* v,
                        const double* rhs, double* x, int lanes, int blocks, int absent,
                        uint64_t wait_ns, double rtol, int max_iter, int32_t* out, double* res) {
  using fs::CgCtl;
  if (blocks < 1 || blocks > fs::kCgMaxBlocks) return -1;
  Pool P;
  std::vector<double> zero(n, 0.0), dinv(n, 0.0), part(9 * fs::kCgMaxBlocks, 0.0);
  for (int64_t r = 0; r < n; ++r)
    for (int32_t k = rp[r]; k < rp[r + 1]; ++k)
      if (ci[k] == r) dinv[r] = 1.0 / v[k];
  std::vector<uint8_t> fixed(n, 0);
  fs::CgOp op;
  op.n = n;
  op.fixed = P.up(fixed.data(), n);
  op.rp = P.up(rp, n + 1);
  op.ci = P.up(ci, rp[n]);
  op.v = P.up(v, rp[n]);
  CgCtl c{};
  c.bar = 0u - (unsigned)absent;
  double* dx = P.up(x, n);
  const double *db = P.up(rhs, n), *dd = P.up(dinv.data(), n);
  double *r = P.up(zero.data(), n), *z = P.up(zero.data(), n), *p = P.up(zero.data(), n),
         *p2 = P.up(zero.data(), n), *q = P.up(zero.data(), n), *dp = P.up(part.data(), part.size());
  CgCtl* dc = P.up(&c, 1);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(128);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  auto k = lanes == 8 ? fs::k_cg_solve<1, 8> : fs::k_cg_solve<1, 1>;
  if (cudaLaunchKernelEx(&cfg, k, op, db, dx, dd, r, z, p, p2, q, dp, dc, rtol, max_iter,
                         wait_ns) != cudaSuccess)
    return -2;
  if (cudaDeviceSynchronize() != cudaSuccess) return -3;
  cudaMemcpy(x, dx, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaMemcpy(&c, dc, sizeof(c), cudaMemcpyDeviceToHost);
  out[0] = c.iters;
  out[1] = c.bad;
  res[0] = c.rr;
  res[1] = c.bb;
  return 0;
}
