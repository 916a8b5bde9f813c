// FP64 block linear algebra and the Round-step kernels (Algorithm 3).
//
//  * k_chol_inv   -- Cholesky of c SPD d x d blocks (one CTA per block, in registers),
//                    explicit inverse A^{-1} = L^{-T} L^{-1}; a non-positive pivot raises a
//                    device flag (FIRAL_ERR_NOT_SPD) instead of trapping.
//  * k_sym_tri    -- Householder tridiagonal forms, and k_nu_coop, the root nu of eq. 10 from
//                    them (Round's per-pick path).
//  * k_tilde_eig  -- eigenvalues of L^{-1} H L^{-T} (similar to Sigma^{-1/2} H Sigma^{-1/2}):
//                    two in-place triangular solves, Householder tridiagonalisation and
//                    Sturm-sequence bisection (Golub & Van Loan, Sections 8.3 and 8.4).
//  * k_nu         -- the root of sum_j (nu + mu_j)^{-2} = 1 (eq. 10) by bisection.
//  * Round kernels -- eq. 14 scores with a masked argmax, the block update of H, and the
//                    assembly of B_t (Algorithm 3 lines 7-11).
#include <cooperative_groups.h>

#include <algorithm>

#include "firal_internal.cuh"

namespace cg = cooperative_groups;

namespace firal {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum_d(double v, double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum_d(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double r = 0;
  for (int i = 0; i < nw; ++i) r += red[i];
  __syncthreads();
  return r;
}

// ------------------------------------------------------------------------------------------
// Cholesky + inverse of c blocks
// ------------------------------------------------------------------------------------------
// One block per matrix, 16 x 16 threads; thread (ti, tk) holds the lower elements
// (ti + 16 x, tk + 16 y), x >= y, in registers.  Factor and inverse are one elimination: after
// step j the columns up to j hold Y = L^{-1} (rows past j: its partial sums) and the columns
// past j the trailing matrix, so a step is one update a_ik -= l_i v_k of every row past j with
//   v_k = Y_jk (k < j), 1 / L_jj (k = j), l_k (k > j),
// published through shared memory by the owners of row and column j.  The owner of the next
// pivot takes its square root and reciprocal while the other threads still update.  The inverse
// is then Y^T Y from shared memory, each 16-row slab only into the columns it reaches.
// d^3 / 2 FP64 multiply-adds per block at two per SM and cycle bound it (d = 64, c = 1000: 0.22
// of 0.57 ms; the rest is the pivots' latency); the form before it kept the matrix in shared memory, three barriers and a
// serial pivot per column, and dot-product chains of up to d dependent multiply-adds (64 cycles
// each) in the inverse: 883 us there, 590 us at d = 100, c = 101 (now 307), 188 us at
// d = 50, c = 10 (now 80).
template <class T, int R>
__global__ __launch_bounds__(256) void k_chol_inv(const double* __restrict__ A, int d,
                                                  T* __restrict__ inv_t,
                                                  double* __restrict__ inv_d,
                                                  double* __restrict__ L_out, int32_t* not_spd) {
  extern __shared__ double sh[];
  __shared__ double vec[16 * R];
  __shared__ double piv[2];          // L_jj and its reciprocal
  const int k0 = blockIdx.x, tid = threadIdx.x, ti = tid >> 4, tk = tid & 15;
  const double* Ak = A + (int64_t)k0 * d * d;
  double* Lk = L_out ? L_out + (int64_t)k0 * d * d : nullptr;
  double a[R * (R + 1) / 2];         // (x, y) at x (x + 1) / 2 + y
#pragma unroll
  for (int x = 0; x < R; ++x)
#pragma unroll
    for (int y = 0; y <= x; ++y) {
      const int i = ti + 16 * x, k = tk + 16 * y;
      a[x * (x + 1) / 2 + y] = i < d && k < d ? Ak[(int64_t)i * d + k] : (i == k ? 1.0 : 0.0);
    }
  if (Lk)
    for (int i = ti; i < d; i += 16)
      for (int k = tk; k < d; k += 16)
        if (k > i) Lk[(int64_t)i * d + k] = 0.0;
  auto pivot = [&](double v) {
    if (!(v > 0.0)) {
      atomicExch(not_spd, 1);
      v = fabs(v) > 1e-300 ? fabs(v) : 1e-300;
    }
    const double r = rsqrt(v);       // a third of the latency of a square root and a division
    piv[0] = v * r;
    piv[1] = r;
  };
  if (tid == 0) pivot(a[0]);
  // steps 16 bj .. 16 bj + 15: bj is a constant, so every register index is one
#pragma unroll
  for (int bj = 0; bj < R; ++bj) {
    const int jn = min(16, d - 16 * bj);
    for (int tj = 0; tj < jn; ++tj) {
      const int j = 16 * bj + tj;
      __syncthreads();               // pivot j is there; the last step's reads of vec are done
      const double r = piv[1];
      if (tk == tj) {                // column j: l_i = a_ij / L_jj, then its column of Y
#pragma unroll
        for (int x = bj; x < R; ++x) {
          const int i = ti + 16 * x;
          double& v = a[x * (x + 1) / 2 + bj];
          if (i > j) {
            const double l = v * r;
            vec[i] = l;
            if (Lk && i < d) Lk[(int64_t)i * d + j] = l;
            v = 0.0;
          } else if (i == j) {
            vec[j] = r;
            if (Lk) Lk[(int64_t)j * d + j] = piv[0];
            v = r;
          }
        }
      }
      if (ti == tj) {                // row j: Y_jk, k < j
#pragma unroll
        for (int y = 0; y <= bj; ++y) {
          const int k = tk + 16 * y;
          double& v = a[bj * (bj + 1) / 2 + y];
          if (k < j) {
            v *= r;
            vec[k] = v;
          }
        }
      }
      __syncthreads();
      // the next pivot first: its square root and reciprocal overlap the update
      if (tj < 15) {
        if (j + 1 < d && ti == tj + 1 && tk == tj + 1) {
          const double l = vec[j + 1];
          pivot(fma(-l, l, a[bj * (bj + 1) / 2 + bj]));
        }
      } else if (bj + 1 < R && j + 1 < d && tid == 0) {
        const double l = vec[j + 1];
        pivot(fma(-l, l, a[bj + 1 < R ? (bj + 1) * (bj + 2) / 2 + bj + 1 : 0]));
      }
      double vk[R];
#pragma unroll
      for (int y = 0; y < R; ++y) vk[y] = vec[tk + 16 * y];
#pragma unroll
      for (int x = bj; x < R; ++x) {
        const int i = ti + 16 * x;
        if (i > j && i < d) {          // (whole warps of padding rows skip)
          const double li = -vec[i];
#pragma unroll
          for (int y = 0; y <= x; ++y)
            a[x * (x + 1) / 2 + y] = fma(li, vk[y], a[x * (x + 1) / 2 + y]);
        }
      }
    }
  }
  if (!inv_t && !inv_d) return;
  // Y to shared memory (zeros above the diagonal)
  const int ld = d | 1;
#pragma unroll
  for (int x = 0; x < R; ++x)
#pragma unroll
    for (int y = 0; y < R; ++y) {
      const int i = ti + 16 * x, k = tk + 16 * y;
      if (i < d && k < d) sh[i * ld + k] = y <= x && k <= i ? a[x * (x + 1) / 2 + (y <= x ? y : 0)] : 0.0;
    }
  __syncthreads();
  // element (p, q) = sum_{i >= p} Y_ip Y_iq, p = ti + 16 x >= 16 x
#pragma unroll
  for (int x = 0; x < R * (R + 1) / 2; ++x) a[x] = 0.0;
#pragma unroll
  for (int s = 0; s < R; ++s) {      // rows 16 s .. 16 s + 15 reach the tiles x <= s
    const int i1 = min(d, 16 * s + 16);
    for (int i = 16 * s; i < i1; ++i) {
      double yk[R], yi[R];
#pragma unroll
      for (int y = 0; y <= s; ++y) {
        yk[y] = tk + 16 * y < d ? sh[i * ld + tk + 16 * y] : 0.0;
        yi[y] = ti + 16 * y < d ? sh[i * ld + ti + 16 * y] : 0.0;
      }
#pragma unroll
      for (int x = 0; x <= s; ++x)
        if (ti + 16 * x < d)
#pragma unroll
          for (int y = 0; y <= x; ++y)
            a[x * (x + 1) / 2 + y] = fma(yi[x], yk[y], a[x * (x + 1) / 2 + y]);
    }
  }
#pragma unroll
  for (int x = 0; x < R; ++x)
#pragma unroll
    for (int y = 0; y <= x; ++y) {
      const int p = ti + 16 * x, q = tk + 16 * y;
      if (p < d && q <= p) {
        const double v = a[x * (x + 1) / 2 + y];
        const int64_t o1 = (int64_t)k0 * d * d + (int64_t)p * d + q;
        const int64_t o2 = (int64_t)k0 * d * d + (int64_t)q * d + p;
        if (inv_t) inv_t[o1] = inv_t[o2] = (T)v;
        if (inv_d) inv_d[o1] = inv_d[o2] = v;
      }
    }
}

static int threads_for(int d) {
  int t = ((d * 2 + 31) / 32) * 32;
  if (t < 64) t = 64;
  if (t > 256) t = 256;
  return t;
}

template <class T, int R>
static int32_t chol_inv_r(const double* A, int c, int d, T* inv_t, double* inv_d, double* L_out,
                          int32_t* not_spd, cudaStream_t st) {
  const size_t smem = (size_t)d * (d | 1) * sizeof(double);
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_chol_inv<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      200 * 1024));
  k_chol_inv<T, R><<<c, 256, inv_t || inv_d ? smem : 0, st>>>(A, d, inv_t, inv_d, L_out, not_spd);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

template <class T>
static int32_t chol_inv_t(const double* A, int c, int d, T* inv_t, double* inv_d, double* L_out,
                          int32_t* not_spd, cudaStream_t st) {
  if (d <= 16) return chol_inv_r<T, 1>(A, c, d, inv_t, inv_d, L_out, not_spd, st);
  if (d <= 32) return chol_inv_r<T, 2>(A, c, d, inv_t, inv_d, L_out, not_spd, st);
  if (d <= 48) return chol_inv_r<T, 3>(A, c, d, inv_t, inv_d, L_out, not_spd, st);
  if (d <= 64) return chol_inv_r<T, 4>(A, c, d, inv_t, inv_d, L_out, not_spd, st);
  if (d <= 96) return chol_inv_r<T, 6>(A, c, d, inv_t, inv_d, L_out, not_spd, st);
  return chol_inv_r<T, 8>(A, c, d, inv_t, inv_d, L_out, not_spd, st);
}

int32_t chol_inv(bool dbl, const double* A, int c, int d, void* inv_t, double* inv_d,
                 double* L_out, int32_t* not_spd, cudaStream_t st) {
  if (d > 128) return fail(FIRAL_ERR_UNSUPPORTED, "block factorisation needs d <= 128");
  ProfScope ps(st, PF_CHOL);
  count_launch();
  if (dbl) return chol_inv_t<double>(A, c, d, (double*)inv_t, inv_d, L_out, not_spd, st);
  return chol_inv_t<float>(A, c, d, (float*)inv_t, inv_d, L_out, not_spd, st);
}

// ------------------------------------------------------------------------------------------
// eigenvalues of L^{-1} H L^{-T}, per block
// ------------------------------------------------------------------------------------------
__device__ int sturm_count(const double* dg, const double* e2, int d, double x) {
  int cnt = 0;
  double q = dg[0] - x;
  if (q < 0) ++cnt;
  for (int i = 1; i < d; ++i) {
    if (q == 0.0) q = 1e-300;
    q = dg[i] - x - e2[i - 1] / q;
    if (q < 0) ++cnt;
  }
  return cnt;
}

// Tridiagonal form of L^{-1} H L^{-T} for one block, in the block's shared memory: the
// similarity (two triangular solves with the reciprocal pivots of L), symmetrisation and
// Householder reduction.  On return dg holds the diagonal and e2 the squared off-diagonal
// (e2[i] couples i and i + 1).  M: d*d doubles; v, p, dg, e2, rl: d doubles each.
__device__ void householder_tridiag(int d, double* M, double* v, double* p, double* dg,
                                    double* e2, double* red);

__device__ void tilde_tridiag(const double* __restrict__ Lk, const double* __restrict__ Hk,
                              int d, double* M, double* v, double* p, double* dg, double* e2,
                              double* rl, double* red) {
  const int tid = threadIdx.x, bd = blockDim.x;
  for (int i = tid; i < d; i += bd) rl[i] = 1.0 / Lk[(int64_t)i * d + i];
  __syncthreads();
  // pass 1: column col of A = L^{-1} H, stored transposed in row col of M
  for (int col = tid; col < d; col += bd) {
    for (int i = 0; i < d; ++i) {
      double acc = Hk[(int64_t)i * d + col];
      for (int q = 0; q < i; ++q) acc -= Lk[(int64_t)i * d + q] * M[col * d + q];
      M[col * d + i] = acc * rl[i];
    }
  }
  __syncthreads();
  // pass 2: column col of M currently holds row col of A; solve L m = that column in place
  for (int col = tid; col < d; col += bd) {
    for (int i = 0; i < d; ++i) {
      double acc = M[i * d + col];
      for (int q = 0; q < i; ++q) acc -= Lk[(int64_t)i * d + q] * M[q * d + col];
      M[i * d + col] = acc * rl[i];
    }
  }
  __syncthreads();
  // symmetrise (rounding)
  for (int t = tid; t < d * d; t += bd) {
    const int i = t / d, j = t % d;
    if (j < i) {
      const double a = 0.5 * (M[i * d + j] + M[j * d + i]);
      M[i * d + j] = a;
      M[j * d + i] = a;
    }
  }
  __syncthreads();
  householder_tridiag(d, M, v, p, dg, e2, red);
}

// Householder reduction of the symmetric d x d matrix M (shared memory, overwritten) to
// tridiagonal form: dg = diagonal, e2 = squared off-diagonal (e2[i] couples i and i + 1).
__device__ void householder_tridiag(int d, double* M, double* v, double* p, double* dg,
                                    double* e2, double* red) {
  const int tid = threadIdx.x, bd = blockDim.x;
  for (int kk = 0; kk + 2 < d; ++kk) {
    double part = 0.0;
    for (int i = kk + 2 + tid; i < d; i += bd) part += M[i * d + kk] * M[i * d + kk];
    const double sigma = block_sum_d(part, red);
    const double x0 = M[(kk + 1) * d + kk];
    if (sigma == 0.0) {
      if (tid == 0) e2[kk] = x0 * x0;
      __syncthreads();
      continue;
    }
    const double mu = sqrt(x0 * x0 + sigma);
    const double alpha = x0 > 0 ? -mu : mu;
    for (int i = kk + 1 + tid; i < d; i += bd) v[i] = i == kk + 1 ? x0 - alpha : M[i * d + kk];
    __syncthreads();
    const double vtv = (x0 - alpha) * (x0 - alpha) + sigma;
    const double tau = 2.0 / vtv;
    for (int i = kk + 1 + tid; i < d; i += bd) {
      double acc = 0.0;
      for (int j = kk + 1; j < d; ++j) acc += M[i * d + j] * v[j];
      p[i] = tau * acc;
    }
    __syncthreads();
    double pv = 0.0;
    for (int i = kk + 1 + tid; i < d; i += bd) pv += p[i] * v[i];
    const double Kc = 0.5 * tau * block_sum_d(pv, red);
    for (int i = kk + 1 + tid; i < d; i += bd) p[i] -= Kc * v[i];   // p becomes w
    __syncthreads();
    const int rem = d - kk - 1;
    for (int t = tid; t < rem * rem; t += bd) {
      const int i = kk + 1 + t / rem, j = kk + 1 + t % rem;
      M[i * d + j] -= v[i] * p[j] + p[i] * v[j];
    }
    if (tid == 0) e2[kk] = alpha * alpha;
    __syncthreads();
  }
  if (tid == 0) {
    if (d >= 2) e2[d - 2] = M[(d - 1) * d + (d - 2)] * M[(d - 1) * d + (d - 2)];
  }
  for (int i = tid; i < d; i += bd) dg[i] = M[i * d + i];
  __syncthreads();
}

__global__ void k_tilde_eig(const double* __restrict__ L, const double* __restrict__ H, int d,
                            double* __restrict__ eig) {
  extern __shared__ double sh[];
  double* M = sh;              // d*d
  double* v = M + d * d;       // d
  double* p = v + d;           // d
  double* dg = p + d;          // d
  double* e2 = dg + d;         // d  (squared off-diagonal)
  double* rl = e2 + d;         // d  (reciprocal pivots of L)
  __shared__ double red[32];
  __shared__ double s_bcast[4];
  const int k = blockIdx.x, tid = threadIdx.x, bd = blockDim.x;
  tilde_tridiag(L + (int64_t)k * d * d, H + (int64_t)k * d * d, d, M, v, p, dg, e2, rl, red);
  // Gershgorin interval (thread 0)
  if (tid == 0) {
    double lo = 1e300, hi = -1e300;
    for (int i = 0; i < d; ++i) {
      const double r = (i > 0 ? sqrt(e2[i - 1]) : 0.0) + (i + 1 < d ? sqrt(e2[i]) : 0.0);
      lo = fmin(lo, dg[i] - r);
      hi = fmax(hi, dg[i] + r);
    }
    const double pad = 1e-12 * fmax(fabs(lo), fabs(hi)) + 1e-300;
    s_bcast[0] = lo - pad;
    s_bcast[1] = hi + pad;
  }
  __syncthreads();
  for (int mth = tid; mth < d; mth += bd) {
    double lo = s_bcast[0], hi = s_bcast[1];
    for (int it = 0; it < 200; ++it) {
      const double mid = 0.5 * (lo + hi);
      if (mid <= lo || mid >= hi) break;
      if (sturm_count(dg, e2, d, mid) > mth) hi = mid;
      else lo = mid;
      if (hi - lo <= 4e-16 * fmax(fabs(lo), fabs(hi))) break;
    }
    eig[(int64_t)k * d + mth] = 0.5 * (lo + hi);
  }
}

// Tridiagonal forms of blocks that are already L^{-1} H L^{-T} (Ht, kept up to date by
// k_round_hupdate): tri[k] = diagonal (d) then squared off-diagonal (d) of block k, gb[k] = its
// Gershgorin interval (lo, hi).  Householder reduction with the matrix in registers: thread
// (ti, tk) of 16 x 16 holds the elements (ti + 16 x, tk + 16 y).  A step publishes its column,
// one warp forms the reflector's scalars, p = tau M v is summed over the 16 threads of a row by
// a butterfly that halves the rows each lane keeps, and M -= v w^T + w v^T runs on registers.
// d^3 FP64 multiply-adds at two per SM and cycle bound it (d = 128: 0.5 ms of 1.05; d = 50:
// 0.03 of 0.22, where the steps' serial part, four barriers, a square root and a division,
// is most).  With the matrix in shared memory and one thread per row of M v, 64 cycles per
// dependent multiply-add, it took 1.77 ms at d = 128, c = 100 and 0.28 ms at d = c = 50.
template <int R>
__global__ __launch_bounds__(256) void k_sym_tri(const double* __restrict__ Ht, int d,
                                                 double* __restrict__ tri,
                                                 double* __restrict__ gb) {
  __shared__ double col[16 * R], w[16 * R], dg[16 * R], e2[16 * R];
  __shared__ double sc[2];           // tau, v_{j+1}
  const int k0 = blockIdx.x, tid = threadIdx.x, ti = tid >> 4, tk = tid & 15, lane = tid & 31;
  const double* Hk = Ht + (int64_t)k0 * d * d;
  double m[R][R];
#pragma unroll
  for (int x = 0; x < R; ++x)
#pragma unroll
    for (int y = 0; y < R; ++y) {
      const int i = ti + 16 * x, k = tk + 16 * y;
      m[x][y] = i < d && k < d ? Hk[(int64_t)i * d + k] : 0.0;
    }
#pragma unroll
  for (int b = 0; b < R; ++b) {
    for (int tj = 0; tj < 16; ++tj) {
      const int j = 16 * b + tj;
      if (j + 2 >= d) break;
      // column j below the diagonal; the diagonal entry is final
      if (tk == tj) {
#pragma unroll
        for (int x = b; x < R; ++x) {
          const int i = ti + 16 * x;
          if (i > j) col[i] = i < d ? m[x][b] : 0.0;
          else if (i == j) dg[j] = m[x][b];
        }
      }
      __syncthreads();
      if (tid < 32) {
        double sg = 0.0;
        for (int i = j + 2 + lane; i < d; i += 32) sg = fma(col[i], col[i], sg);
        sg = warp_sum_d(sg);
        const double x0 = col[j + 1];
        if (lane == 0) {
          if (sg == 0.0) {
            sc[0] = 0.0;
            e2[j] = x0 * x0;
          } else {
            // u = x0 - alpha, |alpha| = mu; u^2 + sg = 2 mu (mu + |x0|), so tau = 1 / (mu |u|)
            const double a2 = fma(x0, x0, sg), r = rsqrt(a2), mu = a2 * r;
            const double u = x0 > 0 ? x0 + mu : x0 - mu;
            sc[0] = r / fabs(u);
            sc[1] = u;
            e2[j] = a2;
          }
        }
      }
      __syncthreads();
      const double tau = sc[0];
      if (tau == 0.0) {
        __syncthreads();             // col and sc are rewritten by the next step
        continue;
      }
      const double u = sc[1];
      double vk[R], vi[R];
#pragma unroll
      for (int y = b; y < R; ++y) {
        const int k = tk + 16 * y, i = ti + 16 * y;
        vk[y] = k <= j ? 0.0 : (k == j + 1 ? u : col[k]);
        vi[y] = i <= j ? 0.0 : (i == j + 1 ? u : col[i]);
      }
      // p = tau M v: row i's 16 partial sums lie in one half-warp
      double ps[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) ps[x] = 0.0;
#pragma unroll
      for (int x = b; x < R; ++x) {
        const int i = ti + 16 * x;
        if (i > j && i < d)            // (whole warps of finished or padding rows skip)
#pragma unroll
          for (int y = b; y < R; ++y) ps[x] = fma(m[x][y], vk[y], ps[x]);
      }
      // lane bits 0, 1, 2 pick which of the 8 rows a lane goes on with; bit 3 adds the halves
#pragma unroll
      for (int h = 4, bit = 1; h >= 1; h >>= 1, bit <<= 1) {
        const bool up = tk & bit;
#pragma unroll
        for (int x = 0; x < h; ++x) {
          const double send = up ? ps[x] : ps[x + h], keep = up ? ps[x + h] : ps[x];
          ps[x] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
        }
      }
      ps[0] += __shfl_xor_sync(0xffffffffu, ps[0], 8);
      if (tk < 8) {
        const int xr = ((tk & 1) << 2) | (tk & 2) | ((tk >> 2) & 1);   // the row this lane kept
        const int i = ti + 16 * xr;
        if (xr < R && i > j) w[i] = tau * ps[0];
      }
      __syncthreads();
      if (tid < 32) {
        double pv = 0.0;
        for (int i = j + 1 + lane; i < d; i += 32)
          pv = fma(w[i], i == j + 1 ? u : col[i], pv);
        pv = warp_sum_d(pv);
        const double K = 0.5 * tau * pv;
        for (int i = j + 1 + lane; i < d; i += 32)      // p becomes w
          w[i] = fma(-K, i == j + 1 ? u : col[i], w[i]);
      }
      __syncthreads();
      double wk[R];
#pragma unroll
      for (int y = b; y < R; ++y) {
        const int k = tk + 16 * y;
        wk[y] = k <= j || k >= d ? 0.0 : w[k];
      }
#pragma unroll
      for (int x = b; x < R; ++x) {
        const int i = ti + 16 * x;
        if (i > j && i < d) {
          const double nv = -vi[x], nw = -w[i];
#pragma unroll
          for (int y = b; y < R; ++y) m[x][y] = fma(nv, wk[y], fma(nw, vk[y], m[x][y]));
        }
      }
    }
  }
  // the last 2 x 2 block (1 x 1 at d = 1)
#pragma unroll
  for (int x = 0; x < R; ++x)
#pragma unroll
    for (int y = 0; y < R; ++y) {
      const int i = ti + 16 * x, k = tk + 16 * y;
      if (i < d && i == k && i + 2 >= d) dg[i] = m[x][y];
      if (i == d - 1 && k == d - 2) e2[d - 2] = m[x][y] * m[x][y];
    }
  __syncthreads();
  for (int i = tid; i < d; i += 256) {
    tri[(int64_t)k0 * 2 * d + i] = dg[i];
    tri[(int64_t)k0 * 2 * d + d + i] = i + 1 < d ? e2[i] : 0.0;
  }
  if (tid < 32) {
    double lo = 1e300, hi = -1e300;
    for (int i = lane; i < d; i += 32) {
      const double r = (i > 0 ? sqrt(e2[i - 1]) : 0.0) + (i + 1 < d ? sqrt(e2[i]) : 0.0);
      lo = fmin(lo, dg[i] - r);
      hi = fmax(hi, dg[i] + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      gb[2 * k0] = lo;
      gb[2 * k0 + 1] = hi;
    }
  }
}

// out_k = L_k^{-1} H_k L_k^{-T} (symmetrised), one block per k
__global__ void k_similarity(const double* __restrict__ L, const double* __restrict__ H, int d,
                             double* __restrict__ out) {
  extern __shared__ double sh[];
  double* M = sh;
  double* rl = M + d * d;
  const int k = blockIdx.x, tid = threadIdx.x, bd = blockDim.x;
  const double* Lk = L + (int64_t)k * d * d;
  const double* Hk = H + (int64_t)k * d * d;
  for (int i = tid; i < d; i += bd) rl[i] = 1.0 / Lk[(int64_t)i * d + i];
  __syncthreads();
  for (int col = tid; col < d; col += bd) {
    for (int i = 0; i < d; ++i) {
      double acc = Hk[(int64_t)i * d + col];
      for (int q = 0; q < i; ++q) acc -= Lk[(int64_t)i * d + q] * M[col * d + q];
      M[col * d + i] = acc * rl[i];
    }
  }
  __syncthreads();
  for (int col = tid; col < d; col += bd) {
    for (int i = 0; i < d; ++i) {
      double acc = M[i * d + col];
      for (int q = 0; q < i; ++q) acc -= Lk[(int64_t)i * d + q] * M[q * d + col];
      M[i * d + col] = acc * rl[i];
    }
  }
  __syncthreads();
  for (int t = tid; t < d * d; t += bd) {
    const int i = t / d, j = t % d;
    out[(int64_t)k * d * d + t] = i == j ? M[t] : 0.5 * (M[i * d + j] + M[j * d + i]);
  }
}

// nu of eq. 10 from the c tridiagonal forms: the root of F(nu) = sum_k Tr((nu I + eta T_k)^-2)
// = 1, which is what sum_j (nu + eta lambda_j)^-2 = 1 states, the trace taken without the
// eigenvalues.
//
// For A = nu I + eta T (diagonal dg, squared off-diagonal e2), the leading principal minors
// theta_i of A (the continuants theta_i = a_i theta_{i-1} - b_i theta_{i-2}, a_i = nu + eta dg_i,
// b_i = eta^2 e2_{i-1}) and their nu-derivatives follow the same three-term recurrence, with no
// division (rescaled by 2^-400 or 2^400 as they grow or shrink; only ratios are used).  With
// t_q = theta^(q) / q!, t_q,i = a_i t_q,i-1 + t_{q-1},i-1 - b_i t_q,i-2, and with p, q2, u the
// ratios of the first, second and third derivative of theta to theta at the last minor (theta_d = det A):
//   Tr A^-2 = p^2 - q2,   d/dnu Tr A^-2 = -2 Tr A^-3 = 3 p q2 - 2 p^3 - u.
//
// Newton runs on psi(nu) = F^(-1/2) - 1: a power mean of the nu + eta lambda_j (exponent -2)
// minus 1, increasing, concave and close to linear right of -eta lambda_min, so the iterates
// reach the root in a few steps; they stay inside the bracket [-eta max Gershgorin,
// sqrt(c d) - eta min Gershgorin], and a step that leaves it, or a trial outside the SPD domain
// (a minor that is not positive), bisects instead.
//
// An SM sub-partition takes a warp's FP64 instruction in 64 cycles however few lanes it has, so
// the four recurrences t_0..t_3 of a class lie in four lanes (two multiply-adds a step, the
// neighbour's term by shuffle) and a warp runs eight classes; a_i is formed by all threads
// before each evaluation.  Blocks of four warps, one grid barrier per step (partials double-
// buffered by step parity; every block takes the same step from them).  c = 100, d = 128:
// 0.29 ms a call, 1.6 ms with one lane per class and 14 FP64 instructions a step; c = d = 50:
// 0.11, 0.58 ms before.
// part: 2 x 3 doubles per block; nu0: a first iterate (taken when inside the bracket) or NULL.
constexpr int NU_CLASSES = 32;   // classes per block

__global__ __launch_bounds__(128) void k_nu_coop(const double* __restrict__ tri,
                                                 const double* __restrict__ gb, int c, int d,
                                                 double eta, const double* nu0, double* part,
                                                 double* nu_out) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ double sh[];
  __shared__ double red[3][4], st[4];   // lo, hi, nu, done
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int ld = d | 1;
  double* as = sh;                      // [32][ld] a_i
  double* es = as + NU_CLASSES * ld;    // [32][ld] eta dg_i
  double* bs = es + NU_CLASSES * ld;    // [32][ld] -b_i
  const bool once = c <= (int)gridDim.x * NU_CLASSES;   // this block's classes: loaded once
  const int ci = tid >> 2, q = tid & 3; // class of the block, derivative
  const double eta2 = eta * eta;
  {
    double a = 1e300, b = -1e300;
    for (int k = tid; k < c; k += 128) {
      a = fmin(a, gb[2 * k]);
      b = fmax(b, gb[2 * k + 1]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      a = fmin(a, __shfl_xor_sync(0xffffffffu, a, o));
      b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    if (lane == 0) {
      red[0][wid] = a;
      red[1][wid] = b;
    }
    __syncthreads();
    if (tid == 0) {
      for (int x = 1; x < 4; ++x) {
        a = fmin(a, red[0][x]);
        b = fmax(b, red[1][x]);
      }
      st[0] = -eta * b;
      st[1] = sqrt((double)c * d) - eta * a;
      const double n0 = nu0 ? *nu0 : st[1];
      st[2] = n0 > st[0] && n0 < st[1] ? n0 : st[1];
      st[3] = 0.0;
    }
  }
  for (int it = 0; it < 300; ++it) {
    __syncthreads();
    const double nu = st[2];
    double f = 0.0, fp = 0.0, bad = 0.0;
    for (int base = blockIdx.x * NU_CLASSES; base < c; base += gridDim.x * NU_CLASSES) {
      const int nc = min(NU_CLASSES, c - base);
      if (it == 0 || !once) {
        __syncthreads();
        for (int x = wid; x < nc; x += 4) {
          const double* t = tri + (int64_t)(base + x) * 2 * d;
#pragma unroll 4
          for (int i = lane; i < d; i += 32) {
            es[x * ld + i] = eta * t[i];
            bs[x * ld + i] = i > 0 ? -eta2 * t[d + i - 1] : 0.0;
          }
        }
        __syncthreads();
      }
      for (int x = wid; x < nc; x += 4)
        for (int i = lane; i < d; i += 32) as[x * ld + i] = nu + es[x * ld + i];
      __syncthreads();
      const int x = min(ci, nc - 1);    // idle lanes repeat the last class
      double u = q == 0 ? 1.0 : 0.0, v = q == 0 ? as[x * ld] : (q == 1 ? 1.0 : 0.0);
      // sign and exponent of theta by integer tests (no FP64 issue): the sign of every minor in
      // the group's first lane, the exponent every fourth step (a step scales by at most
      // |a_i| + |b_i|, far below 2^150)
      bool ok = __double2hiint(v) > 0;
      auto step = [&](int i) {
        double lower = __shfl_up_sync(0xffffffffu, v, 1, 4);
        if (q == 0) lower = 0.0;
        const double nv = fma(as[x * ld + i], v, fma(bs[x * ld + i], u, lower));
        u = v;
        v = nv;
        const int hi = __double2hiint(v);
        ok = ok && hi > 0 && hi < 0x7ff00000;
      };
      int i = 1;
      for (; i + 3 < d; i += 4) {
        step(i);
        step(i + 1);
        step(i + 2);
        step(i + 3);
        const int ex = __shfl_sync(0xffffffffu, __double2hiint(v), lane & ~3) >> 20 & 0x7ff;
        if (ex > 1023 + 400 || (ex < 1023 - 400 && ex > 0)) {
          const double sc = ex > 1023 ? 0x1p-400 : 0x1p400;
          u *= sc;
          v *= sc;
        }
      }
      for (; i < d; ++i) step(i);
      const double t0 = __shfl_sync(0xffffffffu, v, lane & ~3);
      const double t1 = __shfl_sync(0xffffffffu, v, (lane & ~3) + 1);
      const double t2 = __shfl_sync(0xffffffffu, v, (lane & ~3) + 2);
      const double t3 = __shfl_sync(0xffffffffu, v, (lane & ~3) + 3);
      if (q == 0 && ci < nc) {
        if (ok) {
          const double r = 1.0 / t0;
          const double p = t1 * r, qq = 2.0 * t2 * r, uu = 6.0 * t3 * r;
          f += p * p - qq;
          fp += 3.0 * p * qq - 2.0 * p * p * p - uu;
        } else {
          bad = 1.0;
        }
      }
    }
    f = warp_sum_d(f);
    fp = warp_sum_d(fp);
    bad = warp_sum_d(bad);
    if (lane == 0) {
      red[0][wid] = f;
      red[1][wid] = fp;
      red[2][wid] = bad;
    }
    __syncthreads();
    double* pt = part + (size_t)(it & 1) * 3 * gridDim.x;
    if (tid < 3) {
      double a = 0.0;
      for (int x = 0; x < 4; ++x) a += red[tid][x];
      pt[3 * blockIdx.x + tid] = a;
    }
    grid.sync();
    if (tid == 0) {
      double F = 0.0, FP = 0.0, nbad = 0.0;
      for (int b = 0; b < (int)gridDim.x; ++b) {
        F += __ldcg(pt + 3 * b);
        FP += __ldcg(pt + 3 * b + 1);
        nbad += __ldcg(pt + 3 * b + 2);
      }
      const bool off = nbad > 0.0;
      double lo = st[0], hi = st[1];
      if (off || F - 1.0 > 0.0) lo = nu;   // left of the root, or of the domain
      else hi = nu;
      if (!off && F - 1.0 == 0.0) {
        st[3] = 1.0;
      } else {
        // psi = F^-1/2 - 1, psi' = -F^-3/2 F' / 2: nu - psi / psi' = nu + 2 (F - F^3/2) / F'
        const bool newton = !off && FP < 0.0 && F > 0.0;
        const double step = newton ? 2.0 * (F - F * sqrt(F)) / FP : 0.0;
        // Newton converges quadratically: a step below 1e-12 nu leaves the next one far below
        // the accuracy of F itself (~1e-13, the continuant ratios), so take it and stop
        if (newton && fabs(step) <= 1e-12 * fabs(nu)) {
          st[2] = nu + step;
          st[3] = 1.0;
        } else {
          double nx = newton ? nu + step : 0.5 * (lo + hi);
          if (!(nx > lo && nx < hi)) nx = 0.5 * (lo + hi);
          if (nx == nu || hi - lo <= 4e-16 * fmax(fabs(lo), fabs(hi))) st[3] = 1.0;
          st[2] = nx;
        }
      }
      st[0] = lo;
      st[1] = hi;
    }
    __syncthreads();
    if (st[3] != 0.0) break;
  }
  if (blockIdx.x == 0 && tid == 0) *nu_out = st[2];
}

int32_t sym_tri(const double* Ht, int nblocks, int d, double* tri, double* gb, cudaStream_t st) {
  if (d > 128) return fail(FIRAL_ERR_UNSUPPORTED, "tridiagonal forms need d <= 128");
  ProfScope ps(st, PF_ROUND);
  count_launch();
  if (d <= 16) k_sym_tri<1><<<nblocks, 256, 0, st>>>(Ht, d, tri, gb);
  else if (d <= 32) k_sym_tri<2><<<nblocks, 256, 0, st>>>(Ht, d, tri, gb);
  else if (d <= 64) k_sym_tri<4><<<nblocks, 256, 0, st>>>(Ht, d, tri, gb);
  else if (d <= 96) k_sym_tri<6><<<nblocks, 256, 0, st>>>(Ht, d, tri, gb);
  else k_sym_tri<8><<<nblocks, 256, 0, st>>>(Ht, d, tri, gb);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

// nu from c tridiagonal forms (tri: 2 c d doubles, gb: 2 c) on up to one block per SM;
// part: 6 doubles per SM; nu0 (device) may be NULL.
int32_t nu_of_tri(const double* tri, const double* gb, int c, int d, double eta,
                  const double* nu0, double* part, double* nu_out, cudaStream_t st) {
  ProfScope ps(st, PF_ROUND);
  count_launch();
  int dev = 0, sms = 0;
  FIRAL_CUDA_TRY(cudaGetDevice(&dev));
  FIRAL_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int nb = std::min((c + NU_CLASSES - 1) / NU_CLASSES, sms);
  const size_t smem = (size_t)3 * NU_CLASSES * (d | 1) * sizeof(double);
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_nu_coop, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      128 * 1024));
  void* args[] = {(void*)&tri, (void*)&gb,  (void*)&c,    (void*)&d,
                  (void*)&eta, (void*)&nu0, (void*)&part, (void*)&nu_out};
  FIRAL_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)k_nu_coop, dim3(nb), dim3(128), args,
                                             smem, st));
  return FIRAL_OK;
}

int32_t similarity_blocks(const double* L, const double* H, int c, int d, double* out,
                          cudaStream_t st) {
  const size_t smem = ((size_t)d * d + (size_t)d) * sizeof(double);
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_similarity, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      200 * 1024));
  ProfScope ps(st, PF_ROUND);
  count_launch();
  k_similarity<<<c, threads_for(d), smem, st>>>(L, H, d, out);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

int32_t tilde_eigvals(const double* L, const double* H, int c, int d, double* eig,
                      cudaStream_t st) {
  const size_t smem = ((size_t)d * d + 5 * (size_t)d) * sizeof(double);
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_tilde_eig, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      200 * 1024));
  ProfScope ps(st, PF_ROUND);
  count_launch();
  k_tilde_eig<<<c, threads_for(d), smem, st>>>(L, H, d, eig);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

__global__ void k_identity_blocks(double* L, int64_t total, int d) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i % ((int64_t)d * d);
    L[i] = (r / d == r % d) ? 1.0 : 0.0;
  }
}

int32_t identity_blocks(double* L, int c, int d, cudaStream_t st) {
  const int64_t total = (int64_t)c * d * d;
  count_launch();
  k_identity_blocks<<<(unsigned)std::min<int64_t>((total + 255) / 256, 4096), 256, 0, st>>>(L, total, d);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

// ------------------------------------------------------------------------------------------
// nu of eq. 10: sum_j (nu + scale*lam_j)^{-2} = 1, one block
// ------------------------------------------------------------------------------------------
__global__ void k_nu(const double* lam, int64_t count, double scale, double* nu_out) {
  __shared__ double red[32];
  __shared__ double s_lo, s_hi;
  double mn = 1e300;
  for (int64_t i = threadIdx.x; i < count; i += blockDim.x) mn = fmin(mn, scale * lam[i]);
  // block min
  for (int o = 16; o > 0; o >>= 1) mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mn;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 1e300;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) m = fmin(m, red[i]);
    s_lo = -m;
    s_hi = sqrt((double)count) - m;
  }
  __syncthreads();
  double lo = s_lo, hi = s_hi;
  for (int it = 0; it < 400; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    double part = 0.0;
    for (int64_t i = threadIdx.x; i < count; i += blockDim.x) {
      const double a = mid + scale * lam[i];
      part += 1.0 / (a * a);
    }
    const double f = block_sum_d(part, red) - 1.0;
    if (f > 0) lo = mid;
    else hi = mid;
    if (hi - lo <= 1e-15 * fmax(fabs(hi), 1.0)) break;
  }
  if (threadIdx.x == 0) *nu_out = 0.5 * (lo + hi);
}

int32_t nu_bisect_dev(const double* lam, int64_t count, double scale, double* nu_out,
                      cudaStream_t st) {
  ProfScope ps(st, PF_ROUND);
  count_launch();
  k_nu<<<1, 256, 0, st>>>(lam, count, scale, nu_out);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

// ------------------------------------------------------------------------------------------
// Round kernels
// ------------------------------------------------------------------------------------------
// out = a*X + b*Y + c*Z (elementwise over c*d*d doubles); Y, Z may be null
__global__ void k_axpbypcz(double* out, double a, const double* X, double b, const double* Y,
                           double cc, const double* Z, int64_t total) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    double v = a * X[i];
    if (Y) v += b * Y[i];
    if (Z) v += cc * Z[i];
    out[i] = v;
  }
}

__global__ void k_axpbypcz_nu(double* out, const double* nu, const double* X, double b,
                              const double* Y, double cc, const double* Z, int64_t total) {
  const double a = *nu;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = a * X[i] + b * Y[i] + cc * Z[i];
}

// M1_k = Binv_k Sig_k Binv_k (double in, T out); M2_k = Binv_k as T.  Binv_k sits in shared
// memory; Sig_k Binv_k goes through the global scratch Tg (c*d*d doubles).
template <class T>
__global__ void k_round_m(const double* __restrict__ Binv, const double* __restrict__ Sig, int d,
                          T* __restrict__ M1, T* __restrict__ M2, double* __restrict__ Tg,
                          int c_sig) {
  extern __shared__ double sh[];
  double* Bs = sh;           // d*d
  const int k = blockIdx.x, tid = threadIdx.x, bd = blockDim.x;
  const double* Bk = Binv + (int64_t)k * d * d;
  const double* Sk = Sig + (int64_t)(k % c_sig) * d * d;   // Sigma shared by stacked chains
  double* Ts = Tg + (int64_t)k * d * d;
  for (int t = tid; t < d * d; t += bd) Bs[t] = Bk[t];
  __syncthreads();
  for (int t = tid; t < d * d; t += bd) {
    const int i = t / d, j = t % d;
    double acc = 0.0;
    for (int q = 0; q < d; ++q) acc += Sk[(int64_t)i * d + q] * Bs[q * d + j];
    Ts[t] = acc;
  }
  __syncthreads();
  for (int t = tid; t < d * d; t += bd) {
    const int i = t / d, j = t % d;
    double acc = 0.0;
    for (int q = 0; q < d; ++q) acc += Bs[i * d + q] * Ts[q * d + j];
    M1[(int64_t)k * d * d + t] = (T)acc;
    M2[(int64_t)k * d * d + t] = (T)Bs[t];
  }
}

// The same for f32 outputs, in f32 arithmetic.  The consumers keep at most f32 (the SIMT
// scores) or bf16 hi + lo (2^-17 per entry, the tensor-core scores) of M1 and M2, and an f32
// product over d terms carries about sqrt(d) 2^-24 of its row norms, so the FP64 products
// (2 d^3 FMAs per block on a part whose FP64 rate is a small fraction of its FP32 rate) buy
// nothing the picks can use.  Binv_k, Sig_k Binv_k and (when it fits) Sig_k in shared memory.
__global__ void k_round_m_f32(const double* __restrict__ Binv, const double* __restrict__ Sig,
                              int d, float* __restrict__ M1, float* __restrict__ M2, int c_sig,
                              int stage_sig) {
  extern __shared__ float shf[];
  float* Bs = shf;               // d*d
  float* Ts = shf + d * d;       // d*d
  float* Ss = shf + 2 * d * d;   // d*d when stage_sig
  const int k = blockIdx.x, tid = threadIdx.x, bd = blockDim.x;
  const double* Bk = Binv + (int64_t)k * d * d;
  const double* Sk = Sig + (int64_t)(k % c_sig) * d * d;   // Sigma shared by stacked chains
  for (int t = tid; t < d * d; t += bd) {
    const float b = (float)Bk[t];
    Bs[t] = b;
    M2[(int64_t)k * d * d + t] = b;
    if (stage_sig) Ss[t] = (float)Sk[t];
  }
  __syncthreads();
  for (int t = tid; t < d * d; t += bd) {
    const int i = t / d, j = t - i * d;
    float acc = 0.0f;
    if (stage_sig)
      for (int q = 0; q < d; ++q) acc = fmaf(Ss[i * d + q], Bs[q * d + j], acc);
    else
      for (int q = 0; q < d; ++q) acc = fmaf((float)Sk[(int64_t)i * d + q], Bs[q * d + j], acc);
    Ts[t] = acc;
  }
  __syncthreads();
  for (int t = tid; t < d * d; t += bd) {
    const int i = t / d, j = t - i * d;
    float acc = 0.0f;
    for (int q = 0; q < d; ++q) acc = fmaf(Bs[i * d + q], Ts[q * d + j], acc);
    M1[(int64_t)k * d * d + t] = acc;
  }
}

// H_k += H_o,k / b + w_ik x_i x_i^T for the pick i (Algorithm 3 line 8; pool row i read from
// the device, w_ik = h_ik (1 - h_ik)); with L and Ht given,
// the transformed blocks too: Ht_k += Hot_k / b + w_ik y y^T with y = L_k^{-1} x_i
// (Hot = L^{-1} H_o L^{-T}), so that Ht stays L^{-1} H L^{-T} without a similarity per pick.
// Dynamic shared memory: d doubles (with L).
template <class T>
__global__ void k_round_hupdate(double* H, const double* Ho, double invb, const T* Xa,
                                const T* Ha, int64_t m, int d, int c, const int32_t* it_ptr,
                                int32_t t_index, const double* L, double* Ht,
                                const double* Hot) {
  extern __shared__ double ys[];
  const int k = blockIdx.x;
  const int64_t row = m + it_ptr[t_index];
  const double hv = (double)Ha[row * c + k];
  const double wk = hv * (1.0 - hv);
  for (int t = threadIdx.x; t < d * d; t += blockDim.x) {
    const int e = t / d, f = t % d;
    const double xe = (double)Xa[row * d + e], xf = (double)Xa[row * d + f];
    H[(int64_t)k * d * d + t] += Ho[(int64_t)k * d * d + t] * invb + wk * xe * xf;
  }
  if (!L) return;
  // y = L_k^{-1} x: forward substitution, column by column
  const double* Lk = L + (int64_t)k * d * d;
  for (int e = threadIdx.x; e < d; e += blockDim.x) ys[e] = (double)Xa[row * d + e];
  __syncthreads();
  for (int q = 0; q < d; ++q) {
    const double yq = ys[q] / Lk[(int64_t)q * d + q];
    __syncthreads();
    if (threadIdx.x == 0) ys[q] = yq;
    for (int i = q + 1 + threadIdx.x; i < d; i += blockDim.x) ys[i] -= Lk[(int64_t)i * d + q] * yq;
    __syncthreads();
  }
  for (int t = threadIdx.x; t < d * d; t += blockDim.x) {
    const int e = t / d, f = t % d;
    Ht[(int64_t)k * d * d + t] += Hot[(int64_t)k * d * d + t] * invb + wk * ys[e] * ys[f];
  }
}

// eq. 14 scores for pool rows, masked argmax partial per block
template <class T>
__global__ __launch_bounds__(128) void k_round_scores(const T* __restrict__ Xa,
                                                      const T* __restrict__ HaT,
                                                      const T* __restrict__ M1,
                                                      const T* __restrict__ M2,
                                                      const uint8_t* __restrict__ mask,
                                                      int64_t m, int64_t N, int d, int c,
                                                      double eta, double* part_val,
                                                      int64_t* part_idx) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* xs = (T*)smem_raw;           // [d][128]
  T* Ms = xs + (size_t)d * 128;   // d*d
  __shared__ double bv[4];
  __shared__ int64_t bi[4];
  const int tid = threadIdx.x;
  const int64_t r0 = m + (int64_t)blockIdx.x * 128;
  const int64_t row = r0 + tid;
  for (int idx = tid; idx < d * 128; idx += 128) {
    const int r = idx / d, e = idx - r * d;
    const int64_t ii = r0 + r;
    xs[e * 128 + r] = ii < N ? Xa[ii * d + e] : T(0);
  }
  double score = 0.0;
  for (int k = 0; k < c; ++k) {
    double q[2];
    for (int which = 0; which < 2; ++which) {
      const T* Mk = (which == 0 ? M1 : M2) + (int64_t)k * d * d;
      __syncthreads();
      for (int t = tid; t < d * d; t += 128) Ms[t] = Mk[t];
      __syncthreads();
      double acc = 0.0;
      for (int e0 = 0; e0 < d; e0 += 16) {
        T y[16];
#pragma unroll
        for (int ee = 0; ee < 16; ++ee) y[ee] = T(0);
        for (int f = 0; f < d; ++f) {
          const T xf = xs[f * 128 + tid];
#pragma unroll
          for (int ee = 0; ee < 16; ++ee)
            if (e0 + ee < d) y[ee] = fma(Ms[f * d + e0 + ee], xf, y[ee]);   // M symmetric
        }
#pragma unroll
        for (int ee = 0; ee < 16; ++ee)
          if (e0 + ee < d) acc += (double)y[ee] * (double)xs[(e0 + ee) * 128 + tid];
      }
      q[which] = acc;
    }
    if (row < N) {
      const double hv = (double)HaT[(int64_t)k * N + row];
      const double wk = hv * (1.0 - hv);
      score += wk * q[0] / (1.0 + eta * wk * q[1]);
    }
  }
  double val = -INFINITY;
  int64_t idx = INT64_MAX;
  if (row < N && !mask[row - m] && score == score) {
    val = score;
    idx = row - m;
  }
  // block argmax, lowest index on ties
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, val, o);
    const int64_t oi = __shfl_xor_sync(0xffffffffu, idx, o);
    if (ov > val || (ov == val && oi < idx)) {
      val = ov;
      idx = oi;
    }
  }
  if ((tid & 31) == 0) {
    bv[tid >> 5] = val;
    bi[tid >> 5] = idx;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 4; ++w)
      if (bv[w] > val || (bv[w] == val && bi[w] < idx)) {
        val = bv[w];
        idx = bi[w];
      }
    part_val[blockIdx.x] = val;
    part_idx[blockIdx.x] = idx;
  }
}

__global__ void k_round_pick(const double* part_val, const int64_t* part_idx, int np,
                             uint8_t* mask, int32_t* sel, int32_t t, double* score_out) {
  __shared__ double bv[32];
  __shared__ int64_t bi[32];
  double val = -INFINITY;
  int64_t idx = INT64_MAX;
  for (int i = threadIdx.x; i < np; i += blockDim.x) {
    const double v = part_val[i];
    const int64_t ix = part_idx[i];
    if (v > val || (v == val && ix < idx)) {
      val = v;
      idx = ix;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, val, o);
    const int64_t oi = __shfl_xor_sync(0xffffffffu, idx, o);
    if (ov > val || (ov == val && oi < idx)) {
      val = ov;
      idx = oi;
    }
  }
  if ((threadIdx.x & 31) == 0) {
    bv[threadIdx.x >> 5] = val;
    bi[threadIdx.x >> 5] = idx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      if (bv[w] > val || (bv[w] == val && bi[w] < idx)) {
        val = bv[w];
        idx = bi[w];
      }
    if (idx == INT64_MAX) idx = 0;   // nothing selectable (caller validated budget <= n)
    sel[t] = (int32_t)idx;
    mask[idx] = 1;
    *score_out = val;
  }
}

template <class T>
static int32_t round_scores_t(firal_problem* P, const void* M1, const void* M2,
                              const uint8_t* mask, double eta, double* pv, int64_t* pi, int np) {
  const int d = P->d;
  const size_t smem = ((size_t)d * 128 + (size_t)d * d) * sizeof(T);
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_round_scores<T>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  ProfScope ps(P->H->stream, PF_ROUND);
  count_launch();
  k_round_scores<T><<<np, 128, smem, P->H->stream>>>(P->Xa.as<T>(), P->HaT.as<T>(), (const T*)M1,
                                                     (const T*)M2, mask, P->m, P->N, d, P->c, eta,
                                                     pv, pi);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

int32_t round_scores(firal_problem* P, const void* M1, const void* M2, const uint8_t* mask,
                     double eta, double* pv, int64_t* pi, int np) {
  if (!P->dbl)
    return round_scores_f32(P, (const float*)M1, (const float*)M2, mask, eta, pv, pi, np);
  FIRAL_TRY(class_major_h(P));
  return round_scores_t<double>(P, M1, M2, mask, eta, pv, pi, np);
}

int32_t round_pick(const double* pv, const int64_t* pi, int np, uint8_t* mask, int32_t* sel,
                   int32_t t, double* score_out, cudaStream_t st) {
  ProfScope ps(st, PF_ROUND);
  count_launch();
  k_round_pick<<<1, 256, 0, st>>>(pv, pi, np, mask, sel, t, score_out);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

int32_t round_m(bool dbl, const double* Binv, const double* Sig, int c, int d, void* M1, void* M2,
                double* Tg, cudaStream_t st, int n_chain) {
  const size_t smem = (size_t)d * d * sizeof(double);
  const int nb = c * n_chain;   // chains stacked: block k uses Sigma block k mod c
  ProfScope ps(st, PF_ROUND);
  count_launch();
  if (dbl) {
    FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_round_m<double>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    k_round_m<double><<<nb, threads_for(d), smem, st>>>(Binv, Sig, d, (double*)M1, (double*)M2,
                                                        Tg, c);
  } else {
    const int stage_sig = (size_t)3 * d * d * sizeof(float) <= 200 * 1024 ? 1 : 0;
    const size_t smem_f = (size_t)(2 + stage_sig) * d * d * sizeof(float);
    FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_round_m_f32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        200 * 1024));
    k_round_m_f32<<<nb, 256, smem_f, st>>>(Binv, Sig, d, (float*)M1, (float*)M2, c, stage_sig);
  }
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

int32_t round_hupdate(firal_problem* P, double* H, const double* Ho, double invb,
                      const int32_t* sel, int32_t t, const double* L, double* Ht,
                      const double* Hot) {
  cudaStream_t st = P->H->stream;
  ProfScope ps(st, PF_ROUND);
  count_launch();
  const size_t smem = (size_t)P->d * sizeof(double);
  if (P->dbl)
    k_round_hupdate<double><<<P->c, 256, smem, st>>>(H, Ho, invb, P->Xa.as<double>(),
                                                     P->Ha.as<double>(), P->m, P->d, P->c, sel,
                                                     t, L, Ht, Hot);
  else
    k_round_hupdate<float><<<P->c, 256, smem, st>>>(H, Ho, invb, P->Xa.as<float>(),
                                                    P->Ha.as<float>(), P->m, P->d, P->c, sel,
                                                    t, L, Ht, Hot);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

int32_t lincomb(double* out, double a, const double* X, double b, const double* Y, double cc,
                const double* Z, int64_t total, cudaStream_t st) {
  ProfScope ps(st, PF_ROUND);
  count_launch();
  k_axpbypcz<<<(unsigned)((total + 255) / 256 > 4096 ? 4096 : (total + 255) / 256), 256, 0, st>>>(
      out, a, X, b, Y, cc, Z, total);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

int32_t lincomb_nu(double* out, const double* nu, const double* X, double b, const double* Y,
                   double cc, const double* Z, int64_t total, cudaStream_t st) {
  ProfScope ps(st, PF_ROUND);
  count_launch();
  k_axpbypcz_nu<<<(unsigned)((total + 255) / 256 > 4096 ? 4096 : (total + 255) / 256), 256, 0,
                  st>>>(out, nu, X, b, Y, cc, Z, total);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

}  // namespace firal
