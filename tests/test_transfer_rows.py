"""The row functions of the grid transfers, compiled for the host (no GPU): every coarse and fine DoF of a small 2D and 3D
pair against plain nested sums, with empty 1D rows (nodes on Dirichlet faces) along every axis,
and with an infinity or NaN among the inputs (it reaches the sums it belongs to, as itself, and no others)."""
import subprocess

import pytest

from paper_2205_15770_gb300 import build as B

PROGRAM = r"""
#include "vec.cuh"
template <bool COH, typename T>
__host__ __device__ T plain_load(const T *p) { return *p; }
#define ld_in plain_load
#undef __device__
#define __device__ __location__(host) __location__(device)
#include "transfer.cuh"
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
using namespace smf;
static std::mt19937 rng(3);
struct Rows {
  std::vector<int> cnt, idx;
  std::vector<double> w;
  Xfer1D<double> view() const { return {cnt.data(), idx.data(), w.data()}; }
};
// n rows of up to `most` distinct nodes below `nodes`; the first and last row empty where `fixed`
static Rows rows(int n, int nodes, int most, int W, bool fixed) {
  Rows r;
  r.cnt.assign(n, 0);
  r.idx.assign(n * W, -1000000);  // past a row: not a node, not a weight
  r.w.assign(n * W, NAN);
  for (int i = 0; i < n; ++i) {
    if (fixed && (i == 0 || i == n - 1)) continue;
    r.cnt[i] = 1 + (int)(rng() % std::min(most, nodes));
    for (int a = 0; a < r.cnt[i]; ++a) {
      r.idx[i * W + a] = (int)((rng() % 2 + 2 * a) % nodes);
      r.w[i * W + a] = (rng() % 2000) / 1000.0 - 0.9995;  // never zero
    }
  }
  return r;
}
template <int W>
static int check(int dim, int k, const int *nc, unsigned fixed_axes, double planted = 0.5) {
  LevelDesc<double> L[2]{};  // coarse, fine
  for (int f = 0; f < 2; ++f) {
    L[f].dim = dim;
    L[f].k = k;
    L[f].nv = L[f].n_p = 1;
    for (int a = 0; a < 3; ++a) {
      const int n = nc[a] << f;
      L[f].N[a] = a < dim ? k * n + 1 : 1;
      L[f].Pn[a] = a < dim ? (k - 1) * n + 1 : 1;
      L[f].nv *= L[f].N[a];
      L[f].n_p *= L[f].Pn[a];
    }
    L[f].n_u = dim * L[f].nv;
  }
  Rows tab[2][2][3];  // [restriction, prolongation][space][axis]
  XferTabs<double> X;
  for (int d = 0; d < 2; ++d)
    for (int sp = 0; sp < 2; ++sp)
      for (int a = 0; a < 3; ++a) {
        const int *from = sp ? L[1 - d].Pn : L[1 - d].N, *to = sp ? L[d].Pn : L[d].N;
        tab[d][sp][a] = rows(to[a], from[a], d ? k + 1 : W, W, !sp && (fixed_axes >> a & 1u));
        (d ? X.p : X.r)[sp][a] = tab[d][sp][a].view();
      }
  int bad = 0;
  for (int d = 0; d < 2; ++d) {
    const LevelDesc<double> &to = L[d], &from = L[1 - d];
    std::vector<double> in(from.n_u + from.n_p), sub(in.size());
    for (double &v : in) v = (rng() % 2000) / 1000.0 - 1.0;
    for (double &v : sub) v = (rng() % 2000) / 1000.0 - 1.0;
    for (int c = 0; c <= dim; ++c) in[c < dim ? c * from.nv + from.nv / 2 : from.n_u + from.n_p / 2] = planted;
    for (long long i = 0; i < to.n_u + to.n_p; ++i) {
      const int sp = i < to.n_u ? 0 : 1;
      const int *N = sp ? to.Pn : to.N, *M = sp ? from.Pn : from.N;
      const long long j = sp ? i - to.n_u : i % to.nv, off = sp ? from.n_u : i / to.nv * from.nv;
      const int g[3] = {(int)(j % N[0]), (int)(j / N[0] % N[1]), (int)(j / N[0] / N[1])};
      const Rows *t = tab[d][sp];
      double s[2] = {};
      for (int c = 0; c < t[2].cnt[g[2]]; ++c)
        for (int b = 0; b < t[1].cnt[g[1]]; ++b)
          for (int a = 0; a < t[0].cnt[g[0]]; ++a) {
            const long long at = off + ((long long)t[2].idx[g[2] * W + c] * M[1] + t[1].idx[g[1] * W + b]) * M[0] + t[0].idx[g[0] * W + a];
            const double w = t[2].w[g[2] * W + c] * t[1].w[g[1] * W + b] * t[0].w[g[0] * W + a];
            s[0] += w * in[at];
            s[1] += w * (in[at] - sub[at]);
          }
      double r[3] = {s[0], s[1], s[1]};
      if (d == 0) {
        r[0] = restrict_terms<double, W, false>(from, to, X, in.data(), nullptr, i, 0, 1);
        r[1] = r[2] = 0.0;
        for (int lane = 0; lane < 8; ++lane) r[1] += restrict_terms<double, W, true>(from, to, X, in.data(), sub.data(), i, lane, 8);
        r[2] = restrict_terms<double, W, true>(from, to, X, in.data(), sub.data(), i, 0, 1);
      } else {
        r[0] = prolong_entry<double, W>(to, from, X, in.data(), i);
      }
      // at most 17^3 terms of at most 2, three products each: 4,913 x 2 x 8 roundings
      for (int q = 0; q < (d ? 1 : 3); ++q) {
        const double e = s[q > 0];
        bad += std::isfinite(e) ? !(std::fabs(r[q] - e) <= 4913 * 2 * 8 * 0x1p-53)
                                : std::isnan(r[q]) != std::isnan(e) || (!std::isnan(e) && r[q] != e);
      }
    }
  }
  if (bad) std::printf("dim %d k %d axes %u: %d rows off\n", dim, k, fixed_axes, bad);
  return bad;
}
int main() {
  const int n2[3] = {2, 1, 1}, n3[3] = {1, 2, 1};
  int bad = 0;
  for (unsigned axes = 0; axes < 8; ++axes) {
    if (axes < 4) bad += check<9>(2, 2, n2, axes) + check<13>(2, 3, n2, axes) + check<17>(2, 4, n2, axes);
    bad += check<9>(3, 2, n3, axes) + check<13>(3, 3, n3, axes);
    for (double v : {(double)INFINITY, -(double)INFINITY, (double)NAN}) bad += check<9>(3, 2, n3, axes, v) + check<13>(3, 3, n3, axes, v);
  }
  return bad ? 1 : 0;
}
"""


def test_rows_on_the_host(tmp_path):
    try:
        nvcc = B.nvcc_path()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "rows.cu", tmp_path / "rows"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-w", *B.ARCH, "-I", B.CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)  # (a negative status: a signal, such as a division by zero)
