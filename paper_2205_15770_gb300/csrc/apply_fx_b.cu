// Fixed-point FP64 cell kernel (k = 2): the full operator, B and B^T, the dispatch and the stored coefficients.
#include "apply_fx.cuh"

namespace smf {
extern template int launch_fx_mode<kApplyA>(const LevelDesc<double> &, const double *, const double *, double *,
                                            double *, const void *, const Fuse<double> *, cudaStream_t, int, long long);
extern template int launch_fx_mode<kApplyA | kApplyBT>(const LevelDesc<double> &, const double *, const double *,
                                                       double *, double *, const void *, const Fuse<double> *,
                                                       cudaStream_t, int, long long);

int launch_cell_apply_fx(const LevelDesc<double> &L, int mode, const double *u, const double *p, double *yu, double *yp,
                         const void *geo, const Fuse<double> *F, cudaStream_t s, int cols, long long ld) {
  if (L.dim != 3 || L.k != 2 || (!L.cartesian && !geo) || L.n_cells >= (1ll << 31)) return -1;
  switch (mode) {
    case kApplyA: return launch_fx_mode<kApplyA>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyBT: return launch_fx_mode<kApplyBT>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyB: return launch_fx_mode<kApplyB>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyA | kApplyBT: return launch_fx_mode<kApplyA | kApplyBT>(L, u, p, yu, yp, geo, F, s, cols, ld);
    case kApplyA | kApplyBT | kApplyB: return launch_fx_mode<kApplyA | kApplyBT | kApplyB>(L, u, p, yu, yp, geo, F, s, cols, ld);
    default: return -1;
  }
}

long long fx_geometry_bytes(long long cells) { return fx_entries(cells) * (long long)sizeof(int2); }

void launch_fx_geometry(const LevelDesc<double> &L, void *out, cudaStream_t s) {
  const long long b = std::min<long long>((L.n_cells + 3) / 4, 152 * 16);
  launch_kernel(k_fx_geometry<2>, dim3((unsigned)b), dim3(128), 0, s, L, static_cast<int2 *>(out));
}
}  // namespace smf
