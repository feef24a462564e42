// FP32 cell kernel of k = 2 with a z plane per thread: launches and the stored coefficients.
#include "apply_pl.cuh"

namespace smf {

int launch_cell_apply_pl(const LevelDesc<float> &L, int mode, const float *u, const float *p, float *yu, float *yp,
                         const void *geo, const Fuse<float> *F, cudaStream_t s, int cols, long long ld) {
  if (L.dim != 3 || L.k != 2 || (!L.cartesian && !geo) || L.n_cells >= (1ll << 31)) return -1;
  switch (mode) {
    case kApplyA: return launch_pl_mode<kApplyA>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyBT: return launch_pl_mode<kApplyBT>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyB: return launch_pl_mode<kApplyB>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyA | kApplyBT: return launch_pl_mode<kApplyA | kApplyBT>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyA | kApplyBT | kApplyB: return launch_pl_mode<kApplyA | kApplyBT | kApplyB>(L, u, p, yu, yp, geo, F, s, cols, ld);
    default: return -1;
  }
}

long long pl_geometry_bytes(long long cells) {
  return (cells + kFxCells - 1) / kFxCells * pl_group_quads() * (long long)sizeof(float4);
}

void launch_pl_geometry(const LevelDesc<double> &L, void *out, cudaStream_t s) {
  const long long b = std::min<long long>((L.n_cells + 3) / 4, 152 * 16);
  launch_kernel(k_pl_geometry<2>, dim3((unsigned)b), dim3(128), 0, s, L, static_cast<float4 *>(out));
}
}  // namespace smf
