// Non-template kernels: SplitMix64 vectors, deterministic FP64 reductions, Gauss-Jordan
// inverse of the (bordered) coarse matrix, and the dense coarse solve.
#include "vec.cuh"

namespace smf {

__global__ void k_splitmix(unsigned long long seed, double *__restrict__ out, long long n) {
  pdl_enter();
  SMF_GRID_LOOP(i, n) out[i] = splitmix64_uniform(seed, i);
}

__global__ void k_mdot_partial(const double *__restrict__ V, long long ldv, int nvec, const double *__restrict__ w,
                               long long n, double *__restrict__ partial) {
  pdl_enter();
  __shared__ double sh[32];
  for (int j = 0; j < nvec; ++j) {
    const double *v = V + (long long)j * ldv;
    double s = 0.0;
    SMF_GRID_LOOP(i, n) s += v[i] * w[i];
    s = block_reduce_sum<double>(s, sh);
    if (threadIdx.x == 0) partial[(long long)j * gridDim.x + blockIdx.x] = s;
  }
}

__global__ void k_sum_partial(const double *__restrict__ a, long long n, double *__restrict__ partial) {
  pdl_enter();
  __shared__ double sh[32];
  double s = 0.0;
  SMF_GRID_LOOP(i, n) s += a[i];
  s = block_reduce_sum<double>(s, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// out[j] = sum_b partial[j*nparts + b]; one block per j
__global__ void k_final_reduce(const double *__restrict__ partial, int nparts, int nvec, double *__restrict__ out) {
  pdl_enter();
  __shared__ double sh[32];
  const int j = blockIdx.x;
  double s = 0.0;
  for (int b = threadIdx.x; b < nparts; b += blockDim.x) s += partial[(long long)j * nparts + b];
  s = block_reduce_sum<double>(s, sh);
  if (threadIdx.x == 0) out[j] = s;
}

__global__ void k_maxpy(const double *__restrict__ V, long long ldv, int nvec, const double *__restrict__ h,
                        double *__restrict__ w, long long n, double sign) {
  pdl_enter();
  SMF_GRID_LOOP(i, n) {
    double s = 0.0;
#pragma unroll 4
    for (int j = 0; j < nvec; ++j) s += h[j] * V[(long long)j * ldv + i];
    w[i] += sign * s;
  }
}

__global__ void k_scale_by_inv_sqrt(const double *__restrict__ w, const double *__restrict__ nrm2,
                                    double *__restrict__ out, long long n) {
  pdl_enter();
  const double s = 1.0 / sqrt(nrm2[0]);
  SMF_GRID_LOOP(i, n) out[i] = s * w[i];
}

__global__ void k_unit(double *__restrict__ e, long long n, long long j) {
  pdl_enter();
  SMF_GRID_LOOP(i, n) e[i] = (i == j) ? 1.0 : 0.0;
}

// Augmented [Kb | I] (row-major nb x 2nb) from the column-major n0 x n0 coarse matrix K0;
// bordered (nb = n0 + 1) with e = (0, 1_p) when `bordered`.
__global__ void k_build_augmented(const double *__restrict__ K0, int n0, long long n_u, int bordered,
                                  double *__restrict__ M) {
  const int nb = n0 + bordered;
  SMF_GRID_LOOP(idx, (long long)nb * 2 * nb) {
    const int i = (int)(idx / (2 * nb)), j = (int)(idx % (2 * nb));
    double v;
    if (j >= nb)
      v = (j - nb == i) ? 1.0 : 0.0;
    else if (i < n0 && j < n0)
      v = K0[(long long)j * n0 + i];
    else if (i == n0 && j == n0)
      v = 0.0;
    else {
      const int other = (i == n0) ? j : i;
      v = other >= n_u ? 1.0 : 0.0;
    }
    M[idx] = v;
  }
}

// Pivot step k of Gauss-Jordan (single block): partial pivoting on column k, row swap,
// row scaling, and the elimination factors fac[i] = M[i][k] (fac[k] = 0).
__global__ void k_gj_pivot(double *__restrict__ M, int nb, int k, double *__restrict__ fac, int *__restrict__ err) {
  __shared__ double bv[1024];
  __shared__ int bi[1024];
  const int ld = 2 * nb;
  double best = -1.0;
  int besti = k;
  for (int i = k + threadIdx.x; i < nb; i += blockDim.x) {
    const double a = fabs(M[(long long)i * ld + k]);
    if (a > best) {
      best = a;
      besti = i;
    }
  }
  bv[threadIdx.x] = best;
  bi[threadIdx.x] = besti;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      if (bv[threadIdx.x + s] > bv[threadIdx.x] ||
          (bv[threadIdx.x + s] == bv[threadIdx.x] && bi[threadIdx.x + s] < bi[threadIdx.x])) {
        bv[threadIdx.x] = bv[threadIdx.x + s];
        bi[threadIdx.x] = bi[threadIdx.x + s];
      }
    }
    __syncthreads();
  }
  const int p = bi[0];
  if (!(bv[0] > 0.0)) {
    if (threadIdx.x == 0) err[0] = 1;
    return;
  }
  if (p != k)
    for (int j = threadIdx.x; j < ld; j += blockDim.x) {
      const double a = M[(long long)k * ld + j];
      M[(long long)k * ld + j] = M[(long long)p * ld + j];
      M[(long long)p * ld + j] = a;
    }
  __syncthreads();
  const double inv = 1.0 / M[(long long)k * ld + k];
  __syncthreads();
  for (int j = threadIdx.x; j < ld; j += blockDim.x) M[(long long)k * ld + j] *= inv;
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += blockDim.x) fac[i] = (i == k) ? 0.0 : M[(long long)i * ld + k];
}

__global__ void k_gj_elim(double *__restrict__ M, int nb, int k, const double *__restrict__ fac) {
  const int ld = 2 * nb;
  const int i = blockIdx.y;
  const double f = fac[i];
  if (f == 0.0) return;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < ld; j += gridDim.x * blockDim.x)
    M[(long long)i * ld + j] -= f * M[(long long)k * ld + j];
}

// One Gauss-Jordan step from M into O, for small matrices: every block finds the pivot of column k itself (its nb
// entries come from L2) and writes its rows of the swapped, scaled and eliminated matrix: one launch a step (7.4 us with
// 403 rows) instead of a single-block pivot kernel and an elimination.  err: a column without a pivot.
__global__ void k_gj_step(const double *__restrict__ M, double *__restrict__ O, int nb, int k, int *__restrict__ err) {
  __shared__ double bv[kVecThreads];
  __shared__ int bi[kVecThreads];
  const int ld = 2 * nb;
  double best = -1.0;
  int besti = k;
  for (int i = k + threadIdx.x; i < nb; i += blockDim.x) {
    const double a = fabs(M[(long long)i * ld + k]);
    if (a > best) {
      best = a;
      besti = i;
    }
  }
  bv[threadIdx.x] = best;
  bi[threadIdx.x] = besti;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s &&
        (bv[threadIdx.x + s] > bv[threadIdx.x] || (bv[threadIdx.x + s] == bv[threadIdx.x] && bi[threadIdx.x + s] < bi[threadIdx.x]))) {
      bv[threadIdx.x] = bv[threadIdx.x + s];
      bi[threadIdx.x] = bi[threadIdx.x + s];
    }
    __syncthreads();
  }
  const int p = bi[0];
  if (!(bv[0] > 0.0) && blockIdx.x == 0 && threadIdx.x == 0) err[0] = 1;
  const double *piv = M + (long long)p * ld;
  const double inv = 1.0 / piv[k];
  for (int i = blockIdx.x; i < nb; i += gridDim.x) {
    double *o = O + (long long)i * ld;
    if (i == k) {
      for (int j = threadIdx.x; j < ld; j += blockDim.x) o[j] = piv[j] * inv;
    } else {
      const double *r = M + (long long)(i == p ? k : i) * ld;
      const double f = r[k];
      for (int j = threadIdx.x; j < ld; j += blockDim.x) o[j] = r[j] - f * (piv[j] * inv);
    }
  }
}

// Kinv (row-major n0 x n0) = top-left block of the right half of M.
__global__ void k_extract_inverse(const double *__restrict__ M, int nb, int n0, double *__restrict__ Kinv) {
  SMF_GRID_LOOP(idx, (long long)n0 * n0) {
    const int i = (int)(idx / n0), j = (int)(idx % n0);
    Kinv[idx] = M[(long long)i * 2 * nb + nb + j];
  }
}

}  // namespace smf

namespace smf {

// The sums over a warp of eight values a lane, value (lane >> 2) in the result: each exchange also halves the values a
// lane still holds, 9 additions instead of the 40 of eight separate reductions (a warp's FP64 addition occupies an
// SM's FP64 unit for 19 clocks).
__device__ __forceinline__ double warp_sum8(double a[8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 4, m = 16; w >= 1; w >>= 1, m >>= 1) {
    const bool hi = lane & m;
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const double send = hi ? a[k] : a[k + w], keep = hi ? a[k + w] : a[k];
      a[k] = keep + __shfl_xor_sync(0xffffffffu, send, m);
    }
  }
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
  return a[0];
}
// h[j] = V_j . w, j < ctl[0] + add, finished by the last block in a fixed order.  Bound by the FP64 unit (a
// multiply-add an entry, 1.8 us a vector of 859,000) and by reading V: eight vectors a pass over w, so that their
// loads are independent, their sums share the reduction, and w is read once for all of them.  (A vector at a time took
// 6.9 us for one and 33 for six.)
__global__ void k_mdot_final_cnt(const double *__restrict__ V, long long ldv, const int *__restrict__ ctl, int add,
                                 const double *__restrict__ w, long long n, double *__restrict__ partial,
                                 unsigned *__restrict__ ticket, double *__restrict__ out) {
  pdl_enter();
  constexpr int NW = kVecThreads / 32;
  __shared__ double sh[NW][8];
  __shared__ int last;
  const int nvec = ctl[0] + add, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j0 = 0; j0 < nvec; j0 += 8) {
    double s[8] = {};
    const double *v = V + (long long)j0 * ldv;
    SMF_GRID_LOOP(i, n) {
      const double wi = w[i];
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (j0 + c < nvec) s[c] += v[c * ldv + i] * wi;
    }
    const double t = warp_sum8(s);
    if ((lane & 3) == 0) sh[warp][lane >> 2] = t;
    __syncthreads();
    if (threadIdx.x < 8 && j0 + (int)threadIdx.x < nvec) {
      double b = 0.0;
#pragma unroll
      for (int k = 0; k < NW; ++k) b += sh[k][threadIdx.x];
      partial[(long long)(j0 + threadIdx.x) * gridDim.x + blockIdx.x] = b;
      __threadfence();  // this block's partial sums before its ticket
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;  // the counter wraps back to 0
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int nparts = gridDim.x;
  for (int j = warp; j < nvec; j += NW) {
    double s = 0.0;
    for (int b = lane; b < nparts; b += 32) s += __ldcg(partial + (long long)j * nparts + b);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[j] = s;
  }
}

__global__ void k_maxpy_cnt(const double *__restrict__ V, long long ldv, const int *__restrict__ ctl, int add,
                            const double *__restrict__ h, double *__restrict__ w, long long n, double sign) {
  pdl_enter();
  const int nvec = ctl[0] + add;
  SMF_GRID_LOOP(i, n) {
    double s = 0.0;
#pragma unroll 4
    for (int j = 0; j < nvec; ++j) s += h[j] * V[(long long)j * ldv + i];
    w[i] += sign * s;
  }
}

// 1 / sqrt(x), by one thread of the block: by all of them the division and the root were the kernel (859,000 entries:
// 24 us on the FP64 unit, for 14 MB).
__device__ __forceinline__ double block_rsqrt(double x) {
  __shared__ double s;
  if (threadIdx.x == 0) s = 1.0 / sqrt(x);
  __syncthreads();
  return s;
}
__global__ void k_scale_to_slot(const double *__restrict__ w, const double *__restrict__ nrm2, double *__restrict__ V,
                                long long ldv, const int *__restrict__ ctl, long long n) {
  pdl_enter();
  const double s = block_rsqrt(nrm2[0]);
  double *out = V + (long long)(ctl[0] + 1) * ldv;
  SMF_GRID_LOOP(i, n) out[i] = s * w[i];
}

__global__ void k_fgmres_givens(KrylovDev K, cudaGraphConditionalHandle cond, int set_cond) {
  pdl_enter();
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  const int m = K.m, j = K.ctl[0];
  double *H = K.H;
  for (int i = 0; i <= j; ++i) H[i * m + j] = K.hcol[i] + K.hcol[(m + 2) + i];
  H[(j + 1) * m + j] = sqrt(K.hcol[2 * (m + 2)]);
  for (int i = 0; i < j; ++i) {
    const double a = H[i * m + j], b = H[(i + 1) * m + j];
    H[i * m + j] = K.cs[i] * a + K.sn[i] * b;
    H[(i + 1) * m + j] = -K.sn[i] * a + K.cs[i] * b;
  }
  const double den = hypot(H[j * m + j], H[(j + 1) * m + j]);
  K.cs[j] = H[j * m + j] / den;
  K.sn[j] = H[(j + 1) * m + j] / den;
  H[j * m + j] = den;
  H[(j + 1) * m + j] = 0.0;
  const double gj = K.g[j];
  K.g[j + 1] = -K.sn[j] * gj;
  K.g[j] = K.cs[j] * gj;
  const int it = K.ctl[1] + 1;
  K.ctl[1] = it;
  K.ctl[0] = j + 1;
  int stop = 0;
  if (!isfinite(K.g[j + 1]))
    stop = 3;
  else if (fabs(K.g[j + 1]) <= K.thresh[0])
    stop = 1;
  else if (it >= K.ctl[3])
    stop = 2;
  else if (j + 1 >= m)
    stop = 4;
  K.ctl[2] = stop;
  if (set_cond) cudaGraphSetConditional(cond, stop == 0 ? 1u : 0u);
}

__global__ void k_fgmres_trisolve(KrylovDev K) {
  pdl_enter();
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  const int m = K.m, jd = K.ctl[0];
  for (int i = jd - 1; i >= 0; --i) {
    double s = K.g[i];
    for (int c = i + 1; c < jd; ++c) s -= K.H[i * m + c] * K.y[c];
    K.y[i] = s / K.H[i * m + i];
  }
}

}  // namespace smf

namespace smf {

__global__ void k_batch_select(const BatchCond B) {
  pdl_enter();
  const int i = threadIdx.x;
  if (blockIdx.x == 0 && i < B.n) {
    const unsigned on = B.ctl[i][2] == 0 ? 1u : 0u;
    cudaGraphSetConditional(B.member[i], on);
    if (B.has_post) cudaGraphSetConditional(B.post[i], on);
  }
}

__global__ void k_batch_any(const BatchCond B) {
  pdl_enter();
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  int any = 0;
  for (int i = 0; i < B.n; ++i) any |= B.ctl[i][2] == 0;
  cudaGraphSetConditional(B.loop, any ? 1u : 0u);
}


}  // namespace smf

namespace smf {

// ---- Lanczos with its coefficients on the device ------------------------------------------------------
// The last block to finish (ticket) adds the blocks' partial sums in a fixed order.
__device__ __forceinline__ void finish_dot(double s, double *sh, double *partial, unsigned *ticket, double *out) {
  __shared__ int last;
  s = block_reduce_sum<double>(s, sh);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = s;
    __threadfence();
    last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) t += __ldcg(partial + b);
  t = block_reduce_sum<double>(t, sh);
  if (threadIdx.x == 0) out[0] = t;
}
// w -= sum_j h_j V_j over j < ctl[0] + add, and nrm2 = w . w in the same pass (finished by the last block).
__global__ void k_maxpy_norm_cnt(const double *__restrict__ V, long long ldv, const int *__restrict__ ctl, int add,
                                 const double *__restrict__ h, double *__restrict__ w, long long n,
                                 double *__restrict__ partial, unsigned *__restrict__ ticket, double *__restrict__ nrm2) {
  pdl_enter();
  __shared__ double sh[32];
  const int nvec = ctl[0] + add;
  double q = 0.0;
  SMF_GRID_LOOP(i, n) {
    double s = 0.0;
#pragma unroll 4
    for (int j = 0; j < nvec; ++j) s += h[j] * V[(long long)j * ldv + i];
    const double x = w[i] - s;
    w[i] = x;
    q += x * x;
  }
  finish_dot(q, sh, partial, ticket, nrm2);
}
__global__ void k_lz_next(const double *__restrict__ w, const double *__restrict__ b2, const double *__restrict__ sq,
                          double *__restrict__ v, double *__restrict__ tmp, long long n) {
  pdl_enter();
  const double s = block_rsqrt(b2[0]);
  SMF_GRID_LOOP(i, n) {
    const double x = s * w[i];
    v[i] = x;
    tmp[i] = sq[i] * x;
  }
}
__global__ void k_lz_w(const double *__restrict__ sq, double *__restrict__ w, const double *__restrict__ vprev,
                       const double *__restrict__ b2prev, const double *__restrict__ v, long long n,
                       double *__restrict__ partial, unsigned *__restrict__ ticket, double *__restrict__ a) {
  pdl_enter();
  __shared__ double sh[32];
  __shared__ double bs;
  if (threadIdx.x == 0) bs = b2prev ? sqrt(b2prev[0]) : 0.0;
  __syncthreads();
  const double b = bs;
  double s = 0.0;
  SMF_GRID_LOOP(i, n) {
    double x = sq[i] * w[i];
    if (b2prev) x -= b * vprev[i];
    w[i] = x;
    s += x * v[i];
  }
  finish_dot(s, sh, partial, ticket, a);
}
__global__ void k_lz_a(const double *__restrict__ a, double *__restrict__ w, const double *__restrict__ v, long long n,
                       double *__restrict__ partial, unsigned *__restrict__ ticket, double *__restrict__ b2) {
  pdl_enter();
  __shared__ double sh[32];
  const double al = a[0];
  double s = 0.0;
  SMF_GRID_LOOP(i, n) {
    const double x = w[i] - al * v[i];
    w[i] = x;
    s += x * x;
  }
  finish_dot(s, sh, partial, ticket, b2);
}

// unit vectors j0 + blockIdx.y as columns ld entries apart
__global__ void k_unit_cols64(double *__restrict__ e, long long n, long long j0, long long ld) {
  SMF_GRID_LOOP(i, n) e[blockIdx.y * ld + i] = i == j0 + blockIdx.y ? 1.0 : 0.0;
}

}  // namespace smf
