// Explicit S~ (schur.cuh): its application with the vector updates around it, and its assembly by probing.
#include "schur.cuh"
#include "vec.cuh"

namespace smf {

// Bound by reading M once (343 entries a row in 3D: 49 MB for 32^3 cells in FP32) on the large levels, by a few load
// latencies on the small ones: 16 us at 32^3 FP32 against about 30 for the launches it replaces, 2.8 at 8^3; 24x16x8
// FP64 6.2 (FP64 unit).  The same tiles through cp.async into shared memory were slower (18 and 8.4 us).  A block takes 32 consecutive rows, a warp one z offset (2D: y
// offset): a lane's 49 entries are coalesced, independent of the vector and loaded before the previous kernel's
// results are waited for; the warp's neighbours (rows +- 3 on 7 lines) are formed once in shared memory instead of
// 49 times from the up to five vectors they are made of.  The seven partial sums are added in a fixed order.
template <typename T, int DIM>
__global__ void __launch_bounds__(32 * kStencilW)
    k_stencil_apply(const T *__restrict__ M, long long ldm, int n, int P0, int P1, const StencilIn<T> in,
                    const StencilOut<T> o, long long ld) {
  constexpr int R = kStencilR, W = kStencilW, LINES = DIM == 3 ? W : 1, E = 32 + 2 * R;
  __shared__ T xs[W][LINES][E], part[W][32];
  const int lane = threadIdx.x, w = threadIdx.y, row0 = blockIdx.x * 32, row = row0 + lane;
  const T *m = M + (long long)w * LINES * W * ldm + row;
  T a[LINES * W];
#pragma unroll
  for (int j = 0; j < LINES * W; ++j) a[j] = __ldg(m + j * ldm);
  pdl_enter();
  const long long cb = blockIdx.y * ld;
  // all of a lane's neighbours at once, a vector at a time: one load latency a vector instead of one a neighbour
  constexpr int NT = (LINES * E + 31) / 32;
  int idx[NT];
  T v[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    const int q = lane + 32 * t, l = q / E, e = q - l * E;
    // (a neighbour off the grid's side is another line's node: its entry is zero)
    const int i = row0 + e - R + (DIM == 3 ? (l - R) * P0 + (w - R) * P0 * P1 : (w - R) * P0);
    idx[t] = q < LINES * E && i >= 0 && i < n ? i : -1;
    v[t] = T(0);
  }
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (k < in.n) {
      const T *vk = in.v[k] + cb;
#pragma unroll
      for (int t = 0; t < NT; ++t)
        if (idx[t] >= 0) v[t] += in.c[k] * vk[idx[t]];
    }
  if (in.d) {
#pragma unroll
    for (int t = 0; t < NT; ++t)
      if (idx[t] >= 0) v[t] *= in.d[idx[t]];
  }
#pragma unroll
  for (int t = 0; t < NT; ++t)
    if (lane + 32 * t < LINES * E) (&xs[w][0][0])[lane + 32 * t] = v[t];
  __syncwarp();
  T s = T(0);
#pragma unroll
  for (int l = 0; l < LINES; ++l)
#pragma unroll
    for (int j = 0; j < W; ++j) s += a[l * W + j] * xs[w][l][lane + j];
  if (!isfinite(s)) {  // zero times an infinity or NaN is not nothing: leave out what lies off the grid
    const int r = row / P0, gx = row - r * P0, gy = r % P1, gz = r / P1, P2 = n / (P0 * P1);
    s = T(0);
    for (int l = 0; l < LINES; ++l) {
      const int y = gy + (DIM == 3 ? l : w) - R, z = DIM == 3 ? gz + w - R : 0;
      for (int j = 0; j < W; ++j) {
        const int x = gx + j - R;
        if (x >= 0 && x < P0 && y >= 0 && y < P1 && z >= 0 && z < P2) s += m[(l * W + j) * ldm] * xs[w][l][lane + j];
      }
    }
  }
  part[w][lane] = s;
  __syncthreads();
  if (w != 0 || row >= n) return;
  s = part[0][lane];
#pragma unroll
  for (int j = 1; j < W; ++j) s += part[j][lane];
  if (o.t) {
    o.t[cb + row] = s;
    return;
  }
  const T x = o.x[cb + row];
  const T f = o.scale * (x + (o.c1 * (o.d ? o.d[cb + row] : x) + o.c2 * o.Dinv[row] * (o.r[cb + row] - s)));
  if (o.out) o.out[cb + row] = f;
  if (o.acc) o.acc[cb + row] += f;
}

template <typename T>
void launch_stencil(const LevelDesc<T> &L, const T *M, const StencilIn<T> &in, const StencilOut<T> &o, int cols,
                    long long ld, cudaStream_t s) {
  const dim3 grid((unsigned)((L.n_p + 31) / 32), (unsigned)cols), block(32, kStencilW);
  const long long ldm = stencil_rows(L.n_p);
  if (L.dim == 3)
    launch_kernel(k_stencil_apply<T, 3>, grid, block, 0, s, M, ldm, (int)L.n_p, L.Pn[0], L.Pn[1], in, o, ld);
  else
    launch_kernel(k_stencil_apply<T, 2>, grid, block, 0, s, M, ldm, (int)L.n_p, L.Pn[0], L.Pn[1], in, o, ld);
}

struct ColourOf {
  int c[3];
};
template <typename T>
__device__ __forceinline__ ColourOf colour_of(const LevelDesc<T> &L, int col) {
  const int px = min(kStencilW, L.Pn[0]), py = min(kStencilW, L.Pn[1]);
  return {{col % px, (col / px) % py, col / (px * py)}};
}
template <typename T>
__device__ __forceinline__ void pressure_node(const LevelDesc<T> &L, int i, int g[3]) {
  const unsigned n0 = (unsigned)L.Pn[0], r = (unsigned)i / n0;
  g[0] = (int)((unsigned)i - r * n0);
  g[1] = (int)(r % (unsigned)L.Pn[1]);
  g[2] = (int)(r / (unsigned)L.Pn[1]);
}
template <typename T>
__global__ void k_stencil_probe(const LevelDesc<T> L, int c0, T *__restrict__ q, long long ld) {
  pdl_enter();
  const ColourOf k = colour_of(L, c0 + (int)blockIdx.y);
  T *qc = q + blockIdx.y * ld;
  SMF_GRID_LOOP(i, L.n_p) {
    int g[3];
    pressure_node(L, (int)i, g);
    bool on = true;
    for (int a = 0; a < L.dim; ++a) on = on && g[a] % kStencilW == k.c[a];
    qc[i] = on ? T(1) : T(0);
  }
}
// w = S~ q on row i is the entry of the one node of the colour within three nodes of i per direction.
template <typename T>
__global__ void k_stencil_store(const LevelDesc<T> L, int c0, const T *__restrict__ w, long long ld, T *__restrict__ M,
                                long long ldm) {
  pdl_enter();
  const ColourOf k = colour_of(L, c0 + (int)blockIdx.y);
  const T *wc = w + blockIdx.y * ld;
  SMF_GRID_LOOP(i, L.n_p) {
    int g[3], o = 0;
    pressure_node(L, (int)i, g);
    bool in = true;
    for (int a = L.dim - 1; a >= 0; --a) {
      const int e = (k.c[a] - g[a] % kStencilW + kStencilR + kStencilW) % kStencilW, j = g[a] + e - kStencilR;
      in = in && j >= 0 && j < L.Pn[a];
      o = o * kStencilW + e;
    }
    if (in) M[o * ldm + i] = wc[i];
  }
}
template <typename T>
void launch_stencil_probe(const LevelDesc<T> &L, int c0, int cols, long long ld, T *q, cudaStream_t s) {
  launch_kernel(k_stencil_probe<T>, dim3(vec_blocks(L.n_p), (unsigned)cols), dim3(kVecThreads), 0, s, L, c0, q, ld);
}
template <typename T>
void launch_stencil_store(const LevelDesc<T> &L, int c0, int cols, long long ld, const T *w, T *M, cudaStream_t s) {
  launch_kernel(k_stencil_store<T>, dim3(vec_blocks(L.n_p), (unsigned)cols), dim3(kVecThreads), 0, s, L, c0, w, ld, M,
                stencil_rows(L.n_p));
}

#define SMF_STENCIL(T)                                                                                                  \
  template void launch_stencil<T>(const LevelDesc<T> &, const T *, const StencilIn<T> &, const StencilOut<T> &, int,  \
                                  long long, cudaStream_t);                                                           \
  template void launch_stencil_probe<T>(const LevelDesc<T> &, int, int, long long, T *, cudaStream_t);                \
  template void launch_stencil_store<T>(const LevelDesc<T> &, int, int, long long, const T *, T *, cudaStream_t);
SMF_STENCIL(float)
SMF_STENCIL(double)

}  // namespace smf
