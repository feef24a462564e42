// 2D cell kernel: one thread per (cell, velocity component), the component's (k+1)^2 nodal tensor in
// registers.  Same operator as stokes_cell_apply (paper Sec. 3.1: K x = sum_tau P_tau K_tau P_tau^T x by sum
// factorisation; Sec. 2 forms a(u,v), b(v,q)), for the Laplacian form with a constant rho.
//
// Bound by the dependency chain of a launch: a 2D level has 10^2 to 10^5 cells, so a launch lasts as long as
// one thread's gather, contractions and scatter.  The point-per-thread kernel passes every 1D contraction
// through shared memory and a block barrier (14 of them for A u, 2.9-7.2 us a launch on 4^2 .. 128^2 cells); here a contraction is a
// register loop against constant-memory tables and there is no barrier.  A warp holds 32 cells of one
// component (coalesced gathers, uniform component), a CTA the two components of 32 cells.
// With the smoother's vector updates folded into the gathers (FUSED, 8 launches a step with k_S = 1 instead of 16) a
// launch takes 3.1-4.1 us at 32^2 .. 128^2 and the FP32 cycle of 128^2 cells 436 us instead of 729.
#pragma once
#include "apply_col.cuh"

namespace smf {

// 1D contractions of a line: values at the Gauss points, collocation derivative there, and the transposes.
// k = 2: the middle Gauss point is the middle node, and the derivative rows are (-3, 4, -1), (-1, 0, 1),
// (1, -4, 3) times one number: 6 operations a line instead of 9.
template <int K, typename T>
struct Line {
  static constexpr int N = K + 1;
  using CT = CTab<T>;
  static __device__ __forceinline__ void values(const T (&in)[N], T (&out)[N]) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if (K == 2 && q == 1) {
        out[1] = in[1];
        continue;
      }
      T s = CT::S(q * N) * in[0];
#pragma unroll
      for (int m = 1; m < N; ++m) s += CT::S(q * N + m) * in[m];
      out[q] = s;
    }
  }
  static __device__ __forceinline__ void values_t(const T (&in)[N], T (&out)[N]) {
#pragma unroll
    for (int m = 0; m < N; ++m) {
      T s = K == 2 ? (m == 1 ? in[1] : T(0)) : CT::S(N + m) * in[1];
      s += CT::S(m) * in[0];
#pragma unroll
      for (int q = 2; q < N; ++q) s += CT::S(q * N + m) * in[q];
      out[m] = s;
    }
  }
  static __device__ __forceinline__ void derivative(const T (&in)[N], T (&out)[N]) {
    if constexpr (K == 2) {
      const T a = CT::D(N + 2), s = in[0] + in[2] - T(2) * in[1], d = a * (in[2] - in[0]), e = T(2) * a;
      out[0] = d - e * s;
      out[1] = d;
      out[2] = d + e * s;
    } else {
#pragma unroll
      for (int q = 0; q < N; ++q) {
        T s = CT::D(q * N) * in[0];
#pragma unroll
        for (int m = 1; m < N; ++m) s += CT::D(q * N + m) * in[m];
        out[q] = s;
      }
    }
  }
  static __device__ __forceinline__ void derivative_t(const T (&in)[N], T (&add)[N]) {
    if constexpr (K == 2) {
      // rows of D^T: (-3, -1, 1), (4, 0, -4), (-1, 1, 3)
      const T a = CT::D(N + 2), d = in[0] - in[2], s = in[0] + in[1] + in[2], a2 = T(2) * a;
      add[0] -= a * s + a2 * (in[0] - in[2]);
      add[1] += T(4) * (a * d);
      add[2] += a * s - a2 * d;
    } else {
#pragma unroll
      for (int m = 0; m < N; ++m)
#pragma unroll
        for (int q = 0; q < N; ++q) add[m] += CT::D(q * N + m) * in[q];
    }
  }
};

template <int K, typename T, int MODE, bool CART, bool FUSED>
__global__ void __launch_bounds__(64)
    stokes_cell_apply_2d(const LevelDesc<T> L, const T *__restrict__ u, const T *__restrict__ p, T *__restrict__ yu,
                         T *__restrict__ yp, const Fuse<T> F, const long long ld) {
  pdl_enter();
  if constexpr (!FUSED) {
    u = column(u, ld);
    p = column(p, ld);
    yu = column(yu, ld);
    yp = column(yp, ld);
  }
  constexpr int N = K + 1, NP = K;
  constexpr bool DO_A = MODE & kApplyA, DO_BT = MODE & kApplyBT, DO_B = MODE & kApplyB;
  constexpr bool NEED_U = DO_A || DO_B;
  using CT = CTab<T>;
  using LN = Line<K, T>;
  const int c = threadIdx.x >> 5;
  const long long cell = (long long)blockIdx.x * 32 + (threadIdx.x & 31);
  if (cell >= L.n_cells) return;
  const int cy = (int)((unsigned)cell / (unsigned)L.n[0]), cx = (int)((unsigned)cell - (unsigned)cy * (unsigned)L.n[0]);
  bool fx[N], fy[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    fx[i] = !((L.faces & 1u) && K * cx + i == 0) && !((L.faces & 2u) && K * cx + i == L.N[0] - 1);
    fy[i] = !((L.faces & 4u) && K * cy + i == 0) && !((L.faces & 8u) && K * cy + i == L.N[1] - 1);
  }
  const long long vbase = c * L.nv + (long long)(K * cy) * L.N[0] + K * cx;
  const long long pbase = (long long)((K - 1) * cy) * L.Pn[0] + (K - 1) * cx;

  // ---- gathers (FUSED: the Fuse combinations; the owner of a node performs the side effects) --------
  T v[N][N];
  if constexpr (FUSED) {
    T raw[kFuseVel + 2][N][N];  // all loads first
    bool own[N][N];
#pragma unroll
    for (int y = 0; y < N; ++y)
#pragma unroll
      for (int x = 0; x < N; ++x) {
        const long long gi = vbase + (long long)y * L.N[0] + x;
        own[y][x] = (x < K || cx == L.n[0] - 1) && (y < K || cy == L.n[1] - 1);
        const bool need = (NEED_U && fx[x] && fy[y]) || (own[y][x] && F.vstore);
        if (F.nv > 0) {
#pragma unroll
          for (int j = 0; j < kFuseVel; ++j) raw[j][y][x] = (need && j < F.nv) ? F.vv[j][gi] : T(0);
          raw[kFuseVel][y][x] = (need && F.vd) ? F.vd[gi] : T(1);
          raw[kFuseVel + 1][y][x] = (need && F.vb) ? F.vb[gi] : T(0);
        } else {
          raw[0][y][x] = need ? u[gi] : T(0);
        }
      }
#pragma unroll
    for (int y = 0; y < N; ++y)
#pragma unroll
      for (int x = 0; x < N; ++x) {
        T val = raw[0][y][x];
        if (F.nv > 0) {
          T s = F.vc[0] * raw[0][y][x];
#pragma unroll
          for (int j = 1; j < kFuseVel; ++j)
            if (j < F.nv) s += F.vc[j] * raw[j][y][x];
          val = raw[kFuseVel + 1][y][x] + raw[kFuseVel][y][x] * s;
        }
        v[y][x] = (fx[x] && fy[y]) ? val : T(0);
        if (own[y][x]) {
          const long long gi = vbase + (long long)y * L.N[0] + x;
          if (F.vstore) F.vstore[gi] = val;
          if (F.vzero[0]) F.vzero[0][gi] = T(0);
          if (F.vzero[1]) F.vzero[1][gi] = T(0);
        }
      }
  } else if (NEED_U) {
#pragma unroll
    for (int y = 0; y < N; ++y)
#pragma unroll
      for (int x = 0; x < N; ++x) v[y][x] = (fx[x] && fy[y]) ? u[vbase + (long long)y * L.N[0] + x] : T(0);
  }
  T pq[N][N];
  if (DO_BT) {
    T pn[NP][NP];
#pragma unroll
    for (int y = 0; y < NP; ++y)
#pragma unroll
      for (int x = 0; x < NP; ++x) {
        const long long gi = pbase + (long long)y * L.Pn[0] + x;
        T val;
        if (FUSED && F.np > 0) {
          T s = T(0);
#pragma unroll
          for (int j = 0; j < kFusePre; ++j)
            if (j < F.np) s += F.pc[j] * F.pv[j][gi];
          val = F.pd[gi] * s;
        } else {
          val = p[gi];
        }
        pn[y][x] = val;
      }
    if constexpr (FUSED) {
      if (c == 0) {
#pragma unroll
        for (int y = 0; y < NP; ++y)
#pragma unroll
          for (int x = 0; x < NP; ++x)
            if ((x < K - 1 || cx == L.n[0] - 1) && (y < K - 1 || cy == L.n[1] - 1)) {
              const long long gi = pbase + (long long)y * L.Pn[0] + x;
              if (F.pacc) F.pacc[gi] += pn[y][x];
#pragma unroll
              for (int j = 0; j < kFusePre; ++j)
                if (F.pzero[j]) F.pzero[j][gi] = T(0);
            }
      }
    }
    T t[NP][N];
#pragma unroll
    for (int y = 0; y < NP; ++y)
#pragma unroll
      for (int q = 0; q < N; ++q) {
        T s = CT::P(q * NP) * pn[y][0];
#pragma unroll
        for (int x = 1; x < NP; ++x) s += CT::P(q * NP + x) * pn[y][x];
        t[y][q] = s;
      }
#pragma unroll
    for (int q = 0; q < N; ++q)
#pragma unroll
      for (int x = 0; x < N; ++x) {
        T s = CT::P(q * NP) * t[0][x];
#pragma unroll
        for (int y = 1; y < NP; ++y) s += CT::P(q * NP + y) * t[y][x];
        pq[q][x] = s;
      }
  }

  // ---- geometry: J column 0 (d/dxi) linear in eta, column 1 (d/deta) linear in xi --------------------
  T e0[2], e1[2], g0[2], g1[2];
  if (!CART) {
    const T *X = L.vert + ((long long)cy * (L.n[0] + 1) + cx) * 2, *Y = X + (long long)(L.n[0] + 1) * 2;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      e0[a] = X[2 + a] - X[a];
      e1[a] = (Y[2 + a] - Y[a]) - e0[a];
      g0[a] = Y[a] - X[a];
      g1[a] = (Y[2 + a] - X[2 + a]) - g0[a];
    }
  }
  const T mu = L.mu_cell ? L.mu_cell[cell] : L.mu;

  // ---- values and reference gradients at the Gauss points ---------------------------------------------
  T gx[N][N], gy[N][N];
  if (NEED_U) {
    T t[N][N];
#pragma unroll
    for (int y = 0; y < N; ++y) LN::values(v[y], t[y]);
#pragma unroll
    for (int x = 0; x < N; ++x) {
      T in[N], out[N];
#pragma unroll
      for (int y = 0; y < N; ++y) in[y] = t[y][x];
      LN::values(in, out);
#pragma unroll
      for (int y = 0; y < N; ++y) v[y][x] = out[y];
      LN::derivative(out, in);
#pragma unroll
      for (int y = 0; y < N; ++y) gy[y][x] = in[y];
    }
#pragma unroll
    for (int y = 0; y < N; ++y) LN::derivative(v[y], gx[y]);
  }
  // ---- point operation: gx, gy become the fluxes, v the value term, qa the pressure test values ------------
  T qa[N][N];
#pragma unroll
  for (int y = 0; y < N; ++y)
#pragma unroll
    for (int x = 0; x < N; ++x) {
      const T w = CT::W(x) * CT::W(y);
      T a00, a01, a10, a11, det;  // adj J
      if (CART) {
        a00 = L.h[1];
        a11 = L.h[0];
        a01 = a10 = T(0);
        det = L.h[0] * L.h[1];
      } else {
        const T xi = CT::W(N + x), eta = CT::W(N + y);
        const T j00 = e0[0] + eta * e1[0], j10 = e0[1] + eta * e1[1], j01 = g0[0] + xi * g1[0], j11 = g0[1] + xi * g1[1];
        a00 = j11;
        a01 = -j01;
        a10 = -j10;
        a11 = j00;
        det = j00 * j11 - j01 * j10;
      }
      // column c of w adj J
      const T k0 = w * (c == 0 ? a00 : a01), k1 = w * (c == 0 ? a10 : a11);
      T f0 = T(0), f1 = T(0);
      if (DO_B) qa[y][x] = -(k0 * gx[y][x] + k1 * gy[y][x]);
      if (DO_A) {
        const T wd = mu * w / det;
        if (CART) {
          f0 = wd * a00 * a00 * gx[y][x];
          f1 = wd * a11 * a11 * gy[y][x];
        } else {
          const T G01 = wd * (a00 * a10 + a01 * a11);
          f0 = wd * (a00 * a00 + a01 * a01) * gx[y][x] + G01 * gy[y][x];
          f1 = G01 * gx[y][x] + wd * (a10 * a10 + a11 * a11) * gy[y][x];
        }
        v[y][x] *= L.gamma_rho * w * det;
      }
      if (DO_BT) {
        f0 -= pq[y][x] * k0;
        f1 -= pq[y][x] * k1;
        if (!DO_A) v[y][x] = T(0);
      }
      if (DO_A || DO_BT) {
        gx[y][x] = f0;
        gy[y][x] = f1;
      }
    }
  // ---- transposed sweeps and scatter ----------------------------------------------------------------------
  if (DO_A || DO_BT) {
#pragma unroll
    for (int y = 0; y < N; ++y) LN::derivative_t(gx[y], v[y]);
    T t[N][N];
#pragma unroll
    for (int x = 0; x < N; ++x) {
      T in[N], out[N];
#pragma unroll
      for (int y = 0; y < N; ++y) {
        in[y] = gy[y][x];
        out[y] = v[y][x];
      }
      LN::derivative_t(in, out);
      LN::values_t(out, in);
#pragma unroll
      for (int y = 0; y < N; ++y) t[y][x] = in[y];
    }
#pragma unroll
    for (int y = 0; y < N; ++y) {
      T out[N];
      LN::values_t(t[y], out);
#pragma unroll
      for (int x = 0; x < N; ++x)
        if (fx[x] && fy[y]) atomicAdd(&yu[vbase + (long long)y * L.N[0] + x], out[x]);
    }
  }
  if (DO_B) {
    T t[NP][N];
#pragma unroll
    for (int b = 0; b < NP; ++b)
#pragma unroll
      for (int x = 0; x < N; ++x) {
        T s = CT::P(b) * qa[0][x];
#pragma unroll
        for (int q = 1; q < N; ++q) s += CT::P(q * NP + b) * qa[q][x];
        t[b][x] = s;
      }
#pragma unroll
    for (int b = 0; b < NP; ++b)
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        T s = CT::P(a) * t[b][0];
#pragma unroll
        for (int q = 1; q < N; ++q) s += CT::P(q * NP + a) * t[b][q];
        atomicAdd(&yp[pbase + (long long)b * L.Pn[0] + a], s);
      }
  }
}

template <int K, typename T, int MODE, bool FUSED>
static int launch_2d_mode(const LevelDesc<T> &L, const T *u, const T *p, T *yu, T *yp, cudaStream_t s, const Fuse<T> &F,
                          int cols, long long ld) {
  const dim3 grid((unsigned)((L.n_cells + 31) / 32), (unsigned)cols), block(64);
  if (L.cartesian)
    launch_kernel(stokes_cell_apply_2d<K, T, MODE, true, FUSED>, grid, block, 0, s, L, u, p, yu, yp, F, ld);
  else
    launch_kernel(stokes_cell_apply_2d<K, T, MODE, false, FUSED>, grid, block, 0, s, L, u, p, yu, yp, F, ld);
  return 0;
}
// A, B^T, B, A + B^T and the full operator; -1 for other modes (mass, symmetric form, unmasked lifting).  cols: plain
// launches on that many vectors at once, ld entries apart.
template <int K, typename T, bool FUSED>
static int launch_2d(const LevelDesc<T> &L, int mode, const T *u, const T *p, T *yu, T *yp, cudaStream_t s,
                     const Fuse<T> &F, int cols = 1, long long ld = 0) {
  switch (mode) {
    case kApplyA: return launch_2d_mode<K, T, kApplyA, FUSED>(L, u, p, yu, yp, s, F, cols, ld);
    case kApplyBT: return launch_2d_mode<K, T, kApplyBT, FUSED>(L, u, p, yu, yp, s, F, cols, ld);
    case kApplyB: return launch_2d_mode<K, T, kApplyB, FUSED>(L, u, p, yu, yp, s, F, cols, ld);
    case kApplyA | kApplyBT: return launch_2d_mode<K, T, kApplyA | kApplyBT, FUSED>(L, u, p, yu, yp, s, F, cols, ld);
    case kApplyA | kApplyBT | kApplyB: return launch_2d_mode<K, T, kApplyA | kApplyBT | kApplyB, FUSED>(L, u, p, yu, yp, s, F, cols, ld);
    default: return -1;
  }
}

}  // namespace smf
