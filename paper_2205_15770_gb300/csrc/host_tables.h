#pragma once
#include <vector>

#include "common.cuh"

namespace smf {
void gauss_legendre01(int n, double *x, double *w);
void gauss_lobatto01(int deg, double *x);
double lagrange(const double *nodes, int n, int i, double x);
double lagrange_deriv(const double *nodes, int n, int i, double x);
void build_tables(int k, Tab1D<double> &t);
void build_transfer(int k, TransferTab<double> &tt);
double tridiag_max_eig(const std::vector<double> &a, const std::vector<double> &b);

template <typename T>
int launch_cell_apply(const LevelDesc<T> &L, const Tab1D<T> *tab, int mode, const T *u, const T *p, T *yu, T *yp,
                      cudaStream_t s, int shape, const T *geo = nullptr, const T *geox = nullptr, const T *rho = nullptr,
                      const GridBarrier *det = nullptr, bool plane = false);
// `cols` vectors at once, ld entries apart
template <int K, typename T>
int launch_cell_apply_cols_k(const LevelDesc<T> &L, const Tab1D<T> *tab, int mode, const T *u, const T *p, T *yu, T *yp,
                             cudaStream_t s, const T *rho, int cols, long long ld);
template <typename T>
int launch_cell_diag(const LevelDesc<T> &L, const Tab1D<T> *tab, T *dAs, T *dSloc, T *dMp, cudaStream_t s,
                     const T *rho, int sym);
template <int K, typename T>
int launch_cell_apply_k(const LevelDesc<T> &L, const Tab1D<T> *tab, int mode, const T *u, const T *p, T *yu, T *yp,
                        cudaStream_t s, int shape, const T *geo, const T *rho);
template <typename T>
int launch_cell_apply_fused(const LevelDesc<T> &L, int mode, const T *u, const T *p, T *yu, T *yp, cudaStream_t s,
                            int shape, const Fuse<T> &F, const T *geo);
template <int K, typename T>
int launch_cell_apply_fused_k(const LevelDesc<T> &L, int mode, const T *u, const T *p, T *yu, T *yp, cudaStream_t s,
                              int shape, const Fuse<T> &F, const T *geo);
template <int K, typename T>
int launch_cell_C_k(const LevelDesc<T> &L, const Tab1D<T> *tab, T cm, T cg, const T *p, T *yp, T sign, T *diag,
                    const T *Ce, cudaStream_t s);
template <int K, typename T>
int launch_cell_C_matrix_k(const LevelDesc<T> &L, const Tab1D<T> *tab, T cm, T cg, T *Ce, cudaStream_t s);
template <int K, typename T>
int launch_col_geometry_k(const LevelDesc<T> &L, T *geo, cudaStream_t s);
template <int K, typename T>
int launch_cell_grad_k(const LevelDesc<T> &L, const Tab1D<T> *tab, const T *u, const T *lam, T *g, cudaStream_t s);
template <int K>
int upload_col_tables(const Tab1D<double> &t, cudaStream_t s);
// Cell-component kernel (launch shape 5, apply_cc.cuh): 3D Cartesian levels with k = 2, 3 (FP32
// and FP64) and trilinear levels with k = 2 (FP32; FP64 where the per-point geometry is stored).
// launch_cell_apply_cc_k returns -1 for a level or mode it does not serve, 0 on a launch, and a
// cudaError_t code when the (deterministic, cooperative) launch fails.
inline bool cc_level_supported(int dim, int k, int cartesian, size_t elt) {
  (void)elt;
  if (dim != 3) return false;
  if (cartesian) return k == 2 || k == 3;
  return k == 2;
}
// The fixed-point FP64 kernel (shape 5, k = 2; plain and, with F, fused launches): -1 for a level or mode
// it does not serve.  geo: trilinear levels, the coefficients that launch_fx_geometry writes at setup
// (fx_geometry_bytes(cells) bytes).
// cols: plain launches on that many vectors at once, ld entries apart.
int launch_cell_apply_fx(const LevelDesc<double> &L, int mode, const double *u, const double *p, double *yu, double *yp,
                         const void *geo, const Fuse<double> *F, cudaStream_t s, int cols = 1, long long ld = 0);
long long fx_geometry_bytes(long long cells);
void launch_fx_geometry(const LevelDesc<double> &L, void *out, cudaStream_t s);
// The FP32 kernel with a z plane per thread (shape 5 with LevelRT::plane, k = 2): as launch_cell_apply_fx.
int launch_cell_apply_pl(const LevelDesc<float> &L, int mode, const float *u, const float *p, float *yu, float *yp,
                         const void *geo, const Fuse<float> *F, cudaStream_t s, int cols = 1, long long ld = 0);
long long pl_geometry_bytes(long long cells);
void launch_pl_geometry(const LevelDesc<double> &L, void *out, cudaStream_t s);
template <int K, typename T>
int launch_cell_apply_cc_k(const LevelDesc<T> &L, int mode, const T *u, const T *p, T *yu, T *yp, const T *geo,
                           const GridBarrier *det, cudaStream_t s);
template <int K>
int upload_cc_tables(const Tab1D<double> &t, cudaStream_t s);
template <int K, typename T>
int launch_cell_apply_cc_fused_k(const LevelDesc<T> &L, int mode, const T *u, const T *p, T *yu, T *yp,
                                 const T *geo, const Fuse<T> &F, cudaStream_t s);
template <int K, typename T>
int launch_cell_diag_k(const LevelDesc<T> &L, const Tab1D<T> *tab, T *dAs, T *dSloc, T *dMp, cudaStream_t s,
                       const T *rho, int sym);
}  // namespace smf
