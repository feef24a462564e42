// S~ = B A^-1_hat B^T of a level as an explicit stencil matrix (k = 2, k_A = 1).
// On the structured grid B^T, A and B couple a pressure node with those at most three cells away per direction, so a
// row has 7^dim entries: M[o][row], o = the neighbour's offset + 3 in base 7 (x fastest), rows padded to a multiple
// of 32 with zeros, entries whose neighbour lies outside the grid zero.
#pragma once
#include "common.cuh"

namespace smf {

constexpr int kStencilR = 3, kStencilW = 2 * kStencilR + 1;

// The vector that S~ is applied to: x = d (sum_i c_i v_i), d = null: 1.
template <typename T>
struct StencilIn {
  const T *d = nullptr;
  const T *v[5] = {};
  T c[5] = {};
  int n = 0;
};
// What becomes of t = S~ x: stored to t, or (t null) the last Chebyshev step dn = c1 (d or x) + c2 Dinv (r - t),
// out = scale (x + dn), acc += out, as k_cheb_step does.
template <typename T>
struct StencilOut {
  T *t = nullptr;
  const T *r = nullptr, *d = nullptr, *x = nullptr, *Dinv = nullptr;
  T c1{}, c2{}, scale{};
  T *out = nullptr, *acc = nullptr;
};

template <typename T>
void launch_stencil(const LevelDesc<T> &L, const T *M, const StencilIn<T> &in, const StencilOut<T> &o, int cols,
                    long long ld, cudaStream_t s);
// Unit probes of the colours c0 .. c0 + cols - 1 (one node in seven per direction) and the entries they give.
inline long long stencil_rows(long long n_p) { return (n_p + 31) / 32 * 32; }
inline int stencil_entries(int dim) { return dim == 3 ? kStencilW * kStencilW * kStencilW : kStencilW * kStencilW; }
template <typename T>
int stencil_colours(const LevelDesc<T> &L) {
  int n = 1;
  for (int a = 0; a < L.dim; ++a) n *= L.Pn[a] < kStencilW ? L.Pn[a] : kStencilW;
  return n;
}
template <typename T>
void launch_stencil_probe(const LevelDesc<T> &L, int c0, int cols, long long ld, T *q, cudaStream_t s);
template <typename T>
void launch_stencil_store(const LevelDesc<T> &L, int c0, int cols, long long ld, const T *w, T *M, cudaStream_t s);

}  // namespace smf
