// 3D cell kernel of Q2-Q1 in FP32 with a z plane per thread (launch shape 5 where the setup's timing prefers it to
// the cell-component kernel): the layout and contractions of apply_fx.cuh (fx_plane) in floating point.
//
// Against the cell-component kernel (27 nodes a thread, geometry evaluated in the kernel): the contractions use
// Q2's tables (6 multiply-adds a line for values, 4-6 operations for derivatives, instead of 9) and the per-point
// coefficients are read (32 bytes a point with an A block, 16 with B or B^T a component), staged in shared memory
// while the values are gathered; a warp's chain is a quarter as long, three times the warps are in flight, and the
// 32^3 level, 1.35 waves of long chains there, fills the GPU with short ones.  Measured (us, cell-component kernel ->
// this kernel, trilinear): 32^3 A 14.4 -> 9.3, B^T 10.5 -> 8.0, B 8.9 -> 6.8, K 20.0 -> 13.7; 16^3 A 7.2 (column
// kernel 5.6) -> 4.4; 8^3 A 5.7 (3.3) -> 2.3.  On Cartesian cells the cell-component kernel's Kronecker form is as
// fast at 32^3 (8.0) and the setup's timing decides.  Bound by latency: at 32^3 issue is half busy, the gathers, the
// staged coefficients and the shuffles take turns.
#pragma once
#include "apply_fx.cuh"

namespace smf {

constexpr int kPlQuads = 5;  // float4 per point: (G00, G01, G02, G11), (G12, G22, W, 0), columns of C
// [group of 10 cells] times a block of the first two and a block of the last three, each [y, x point][quad][lane]
__host__ __device__ inline long long pl_group_quads() { return 9ll * kPlQuads * 32; }

template <int MODE>
struct PlStage {
  static constexpr int G = (MODE & kApplyA) ? 9 * 2 * 32 * (int)sizeof(float4) : 0;
  static constexpr int C = (MODE & (kApplyB | kApplyBT)) ? 9 * 3 * 32 * (int)sizeof(float4) : 0;
};
// Cartesian levels: G (without the viscosity), W and C by weight class (see FxCart).
struct PlCart {
  float g[3][4], w[4], c[3][4];
};
inline PlCart pl_cart(const LevelDesc<float> &L) {
  PlCart K{};
  const double h[3] = {(double)L.h[0], (double)L.h[1], (double)L.h[2]}, v = h[0] * h[1] * h[2];
  for (int m = 0; m < 4; ++m) {
    for (int a = 0; a < 3; ++a) {
      K.g[a][m] = (float)(kFxAlpha2 * v / (h[a] * h[a]) * fx_weight(m));
      K.c[a][m] = (float)(kFxAlpha * v / h[a] * fx_weight(m));
    }
    K.w[m] = (float)(L.gamma_rho * v * fx_weight(m));
  }
  return K;
}

template <int MODE, bool CART, bool FUSED>
__device__ __forceinline__ void pl_group(const LevelDesc<float> &L, const float *__restrict__ u, const float *__restrict__ p,
                                         float *__restrict__ yu, float *__restrict__ yp, const float4 *__restrict__ geo,
                                         long long group, int c, const PlCart &K, const Fuse<float> &F) {
  extern __shared__ int4 fx_smem[];
  using ST = PlStage<MODE>;
  if constexpr (!CART) {
    const float4 *src = geo + group * pl_group_quads();
    plane_stage<ST::G>(src, fx_smem);
    plane_stage<ST::C>(src + 9 * 2 * 32, fx_smem + ST::G / 16);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const PlaneIdx I = plane_index(L, group, c);
  float uv[3][3], pv[2][2][2], qv[2][2];
  plane_gather<MODE, FUSED>(L, I, c, u, p, F, uv, pv);
  FxGeo<FxFlt, CART> g;
  if constexpr (CART) {
    const float mu = L.mu_cell ? L.mu_cell[I.cell] : L.mu;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
#pragma unroll
      for (int a = 0; a < 3; ++a) g.g[a][m] = mu * (I.z == 1 ? K.g[a][m + 1] : K.g[a][m]);
      g.w[m] = I.z == 1 ? K.w[m + 1] : K.w[m];
      g.cc[m] = I.z == 1 ? K.c[c][m + 1] : K.c[c][m];
    }
  } else {
    g.g = reinterpret_cast<const float4 *>(fx_smem) + I.lane;
    g.cc = reinterpret_cast<const float4 *>(fx_smem + ST::G / 16) + I.lane;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  fx_plane<FxFlt, MODE, CART>(uv, pv, qv, g, c, I.z, I.lane, 0);
  plane_scatter<MODE>(I, yu, yp, uv, qv);
}

template <int MODE, bool CART>
__global__ void __launch_bounds__(kFxThreads)
    stokes_cell_apply_pl(const LevelDesc<float> L, const float *__restrict__ u, const float *__restrict__ p,
                         float *__restrict__ yu, float *__restrict__ yp, const float4 *__restrict__ geo, const __grid_constant__ PlCart K,
                         const long long ld) {
  pdl_enter();
  pl_group<MODE, CART, false>(L, column(u, ld), column(p, ld), column(yu, ld), column(yp, ld), geo, blockIdx.x, threadIdx.x >> 5, K, Fuse<float>{});
}
template <int MODE, bool CART>
__global__ void __launch_bounds__(kFxThreads)
    stokes_cell_apply_pl_fused(const LevelDesc<float> L, const float *__restrict__ u, const float *__restrict__ p,
                               float *__restrict__ yu, float *__restrict__ yp, const float4 *__restrict__ geo,
                               const __grid_constant__ PlCart K, const Fuse<float> F) {
  pdl_enter();
  pl_group<MODE, CART, true>(L, u, p, yu, yp, geo, blockIdx.x, threadIdx.x >> 5, K, F);
}

// The coefficients of trilinear cells, formed at setup in FP64 (a warp per cell, a lane per point) and rounded once.
template <int K>
__global__ void k_pl_geometry(const LevelDesc<double> L, float4 *__restrict__ out) {
  pdl_enter();
  const int lane = threadIdx.x & 31, pt = lane < 27 ? lane : 0;
  const int ix = pt % 3, iy = (pt / 3) % 3, iz = pt / 9;
  constexpr double r = 0.38729833462074168852;
  const double xi = 0.5 + (ix - 1) * r, eta = 0.5 + (iy - 1) * r, zeta = 0.5 + (iz - 1) * r;
  const double w = fx_weight((ix == 1) + (iy == 1) + (iz == 1));
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long cell = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); cell < L.n_cells; cell += warps) {
    const int cx = (int)(cell % L.n[0]);
    const long long rr = cell / L.n[0];
    const int cy = (int)(rr % L.n[1]), cz = (int)(rr / L.n[1]);
    double J[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        v[i] = L.vert[(((long long)(cz + (i >> 2)) * (L.n[1] + 1) + (cy + ((i >> 1) & 1))) * (L.n[0] + 1) + (cx + (i & 1))) * 3 + a];
      auto lerp = [](double p, double q, double t) { return p + t * (q - p); };
      J[a][0] = lerp(lerp(v[1] - v[0], v[3] - v[2], eta), lerp(v[5] - v[4], v[7] - v[6], eta), zeta);
      J[a][1] = lerp(lerp(v[2] - v[0], v[3] - v[1], xi), lerp(v[6] - v[4], v[7] - v[5], xi), zeta);
      J[a][2] = lerp(lerp(v[4] - v[0], v[5] - v[1], xi), lerp(v[6] - v[2], v[7] - v[3], xi), eta);
    }
    double adj[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b1 = (b + 1) % 3, b2 = (b + 2) % 3, a1 = (a + 1) % 3, a2 = (a + 2) % 3;
        adj[b][a] = J[a1][b1] * J[a2][b2] - J[a2][b1] * J[a1][b2];
      }
    const double det = J[0][0] * adj[0][0] + J[1][0] * adj[0][1] + J[2][0] * adj[0][2];
    const double wd = kFxAlpha2 * (L.mu_cell ? L.mu_cell[cell] : L.mu) * w / det, wa = kFxAlpha * w;
    auto dot = [&](int i, int j) {
      return (float)(wd * (adj[i][0] * adj[j][0] + adj[i][1] * adj[j][1] + adj[i][2] * adj[j][2]));
    };
    if (lane < 27) {
      float4 *q = out + (cell / kFxCells) * pl_group_quads() + iz * 10 + cell % kFxCells;
      const int yx = lane % 9;
      q[2 * yx * 32] = make_float4(dot(0, 0), dot(0, 1), dot(0, 2), dot(1, 1));
      q[(2 * yx + 1) * 32] = make_float4(dot(1, 2), dot(2, 2), (float)(L.gamma_rho * w * det), 0.f);
#pragma unroll
      for (int c = 0; c < 3; ++c)
        q[(9 * 2 + 3 * yx + c) * 32] = make_float4((float)(wa * adj[0][c]), (float)(wa * adj[1][c]), (float)(wa * adj[2][c]), 0.f);
    }
  }
}

template <int MODE>
static int launch_pl_mode(const LevelDesc<float> &L, const float *u, const float *p, float *yu, float *yp, const void *geo,
                          const Fuse<float> *F, cudaStream_t s, int cols, long long ld) {
  const dim3 grid((unsigned)((L.n_cells + kFxCells - 1) / kFxCells), F ? 1u : (unsigned)cols), block(kFxThreads);
  const float4 *g = static_cast<const float4 *>(geo);
  const PlCart K = L.cartesian ? pl_cart(L) : PlCart{};
  if (F) {
    if (L.cartesian)
      launch_kernel(stokes_cell_apply_pl_fused<MODE, true>, grid, block, 0, s, L, u, p, yu, yp, g, K, *F);
    else
      launch_kernel(stokes_cell_apply_pl_fused<MODE, false>, grid, block, PlStage<MODE>::G + PlStage<MODE>::C, s, L, u, p, yu, yp, g, K, *F);
  } else {
    if (L.cartesian)
      launch_kernel(stokes_cell_apply_pl<MODE, true>, grid, block, 0, s, L, u, p, yu, yp, g, K, ld);
    else
      launch_kernel(stokes_cell_apply_pl<MODE, false>, grid, block, PlStage<MODE>::G + PlStage<MODE>::C, s, L, u, p, yu, yp, g, K,
                    ld);
  }
  return 0;
}

}  // namespace smf
