// Fixed-point FP64 cell kernel (k = 2): the applications with the velocity block alone or with B^T.
#include "apply_fx.cuh"

namespace smf {
template int launch_fx_mode<kApplyA>(const LevelDesc<double> &, const double *, const double *, double *, double *,
                                     const void *, const Fuse<double> *, cudaStream_t, int, long long);
template int launch_fx_mode<kApplyA | kApplyBT>(const LevelDesc<double> &, const double *, const double *, double *,
                                                double *, const void *, const Fuse<double> *, cudaStream_t, int, long long);
}  // namespace smf
