// Drives the solution update of a restart cycle alone (fs_krylov.cu is
// compiled into this file).
#include "fs_krylov.cu"

#include <cstring>
#include <vector>

namespace fs {
void count_launches(int64_t) {}
bool launch_overlap() { return false; }
}  // namespace fs

namespace {

// x (n entries) += Z^T y for the upper triangle H (k x k, row-major) and
// right-hand side g, Z k rows of n entries; tiles of at most kTileLen entries.
template <typename V>
int update(int64_t n, int k, const double* H, const double* g, const double* Z, double* x) {
  const int m = 30;
  std::vector<V> hz(Z, Z + k * n), hx(x, x + n);
  std::vector<fs::Tile> tiles;
  for (int64_t a = 0; a < n; a += fs::kTileLen) {
    fs::Tile t{};
    t.start = a;
    t.len = (int32_t)(n - a < fs::kTileLen ? n - a : fs::kTileLen);
    tiles.push_back(t);
  }
  std::vector<fs::SegState> st(1);
  memset((void*)st.data(), 0, sizeof(fs::SegState));
  st[0].k = k;
  for (int i = 0; i < k; ++i) {
    st[0].g[i] = g[i];
    for (int c = i; c < k; ++c) st[0].H[i * m + c] = H[i * k + c];
  }
  fs::KCtl ctl{};
  ctl.m = m;
  ctl.nseg = 1;
  char* d = nullptr;
  const size_t bz = sizeof(V) * hz.size(), bx = sizeof(V) * hx.size(), bt = sizeof(fs::Tile) * tiles.size();
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t ox = up(bz), ot = ox + up(bx), os = ot + up(bt), oc = os + up(sizeof(fs::SegState));
  if (cudaMalloc((void**)&d, oc + up(sizeof(ctl))) != cudaSuccess) return -1;
  cudaMemcpy(d, hz.data(), bz, cudaMemcpyHostToDevice);
  cudaMemcpy(d + ox, hx.data(), bx, cudaMemcpyHostToDevice);
  cudaMemcpy(d + ot, tiles.data(), bt, cudaMemcpyHostToDevice);
  cudaMemcpy(d + os, st.data(), sizeof(fs::SegState), cudaMemcpyHostToDevice);
  cudaMemcpy(d + oc, &ctl, sizeof(ctl), cudaMemcpyHostToDevice);
  const fs::TileList tl{(const fs::Tile*)(d + ot), (int)tiles.size()};
  fs::launch_seg_update_x<V, V>((const fs::SegState*)(d + os), (const fs::KCtl*)(d + oc),
                                (const V*)d, n, tl, (V*)(d + ox), 0);
  const int rc = cudaDeviceSynchronize() == cudaSuccess ? 0 : -3;
  cudaMemcpy(hx.data(), d + ox, bx, cudaMemcpyDeviceToHost);
  cudaFree(d);
  for (int64_t i = 0; i < n; ++i) x[i] = (double)hx[i];
  return rc;
}

}  // namespace

extern "C" int update_x(int f32, int64_t n, int k, const double* H, const double* g,
                        const double* Z, double* x) {
  return f32 ? update<float>(n, k, H, g, Z, x) : update<double>(n, k, H, g, Z, x);
}
