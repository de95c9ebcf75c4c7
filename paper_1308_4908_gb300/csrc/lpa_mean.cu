// Order 0 with one small window (lpa_mean.cuh): the plain kernels of the smaller windows, the choice of
// a kernel and the launch. The wider windows and the compensated kernels compile beside it
// (lpa_mean_wide.cu, lpa_mean_comp.cu).
#include <cmath>

#include "lpa_dispatch.h"
#include "lpa_mean.cuh"

const void *lpa_mean_wide(const LpaLaunch &L);
const void *lpa_mean_comp(const LpaLaunch &L);

int lpa_mean_size(double reach_rb, double reach_g) {
  const double rb = std::floor(reach_rb) + 1, g = std::floor(reach_g) + 1;
  return rb <= 3 && g <= 2 ? 0 : rb <= 4 && g <= 3 ? 1 : -1;
}
int lpa_mean_cells(int size, bool green) {
  return size >= 2 ? size + 1 : size == 0 ? (green ? 2 : 3) : (green ? 3 : 4);
}
int lpa_mean_k_words(int size) { return size == 0 ? lpa::Layout<3, 2>::kTab : lpa::Layout<4, 3>::kTab; }
int lpa_mean_k_word(int size, int cls, int ph) {
  using A = lpa::Layout<3, 2>;
  using B = lpa::Layout<4, 3>;
  return 16 + (size == 0 ? cls * A::kClass + A::phase_words(ph) : cls * B::kClass + B::phase_words(ph));
}
uint32_t lpa_mean_tab_bytes(int size, bool axis, int classes, bool tab, int p, int n_sensors) {
  if (!axis) return (uint32_t)(n_sensors * lpa_mean_tile_h(p) * 16);
  const int words = size == 0 ? lpa::Layout<3, 2>::kWords : lpa::Layout<4, 3>::kWords;
  const int row = size == 0 ? lpa::Layout<3, 2>::kRow : lpa::Layout<4, 3>::kRow;
  if (tab) return (uint32_t)(n_sensors * 4 * lpa_mean_k_words(size));  // (more than the classes' tables)
  if (classes) return (uint32_t)(n_sensors * 4 * row * classes);
  return (uint32_t)(n_sensors * 4 * (words * lpa::kBW + row * lpa_mean_tile_h(p)));
}
const void *lpa_mean_kernel(const LpaLaunch &L) {
  return L.mean_comp ? lpa_mean_comp(L) : L.mean_size == 0 ? lpa::pick<3, 2, false>(L) : lpa_mean_wide(L);
}
dim3 lpa_mean_grid(const LpaLaunch &L) {
  const int bh = lpa_mean_tile_h(L.mean_p);
  return dim3((unsigned)((L.out_w + lpa::kBW - 1) / lpa::kBW), (unsigned)((L.mean_y1 - L.mean_y0 + bh - 1) / bh));
}
void lpa_mean_rows(LpaLaunch &L, int tile0, int count) {
  L.mean_y0 = tile0 / L.tiles_x * L.tile_h;
  L.mean_y1 = ((tile0 + count - 1) / L.tiles_x + 1) * L.tile_h;
  if (L.mean_y1 > L.out_h) L.mean_y1 = L.out_h;
}
cudaError_t lpa_launch_mean(const LpaLaunch &L, cudaStream_t st) {
  const void *fn = lpa_mean_kernel(L);
  cudaError_t e = lpa_opt_in(fn);
  if (e != cudaSuccess) return e;
  void *args[] = {const_cast<LpaLaunch *>(&L)};
  return cudaLaunchKernel(fn, lpa_mean_grid(L), dim3((unsigned)lpa_mean_threads(L.mean_p)), args, L.smem_bytes, st);
}
