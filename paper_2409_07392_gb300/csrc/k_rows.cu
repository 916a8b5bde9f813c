// Contractions over the rows (points) on the CUDA cores, for FIRAL_FP32 and FIRAL_FP64 and for
// the block sums of Round in every precision:
//
//   k_row_form   per-row forms of x_i.V (f32): the alpha of Lemma 1, the gradient's quadratic
//                forms (eq. 11) and the eq. 14 scores of Round
//   k_row_form_d the first two in FP64
//   k_row_outer  sums over the rows of A[i][m] B[i][n]: the low-rank part of the Hessian apply
//                (m = (probe, class), n = feature), in FP64 also the weighted block sums of
//                eq. 13 (m = class, n = pair of features)
//   k_outer_gemm the f32 block sums and Exact-FIRAL's dense sums, operands written out first
//   k_block_ord  the f32 block sums with every addition in a fixed order
//
// All are dense products.  f32: 8 x 8 or 8 x 16 outputs per thread from shared memory, plain
// fmaf: the packed form (fma.rn.f32x2) has the same peak on this part and needs one operand
// duplicated, which cost more in shared-memory reads than it saved in issue slots (43 against 53
// TFLOP/s with operands resident).  FP64: the part issues two FP64 multiply-adds per SM and
// cycle, so operand traffic is free and what counts is that no lane multiplies padding and every
// SM has work; tiles are 2 x 2 outputs per thread with the tile's width taken from the problem
// instead of a power of two.
#include <cuda_bf16.h>

#include <algorithm>

#include "firal_internal.cuh"

namespace firal {
namespace {

// ------------------------------------------------------------------------------------------
// helpers
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// copies n bytes to shared memory, zeros when !ok (the source address must still be valid)
template <int n>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool ok) {
  const int sz = ok ? n : 0;
  if (n == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
                 "r"(sz)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_addr(dst)), "l"(src),
                 "n"(n), "r"(sz)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ------------------------------------------------------------------------------------------
// k_row_outer: part[split][m][n] = sum over the split's rows of A[i][m] B[i][n]
//   OP 0 (low-rank part):   m = j c + k, A = h_ik walpha_ij; n = e, B = x_ie
//   OP 1 (FP64 block sums): m = which c + k, A = w_i h_ik (which 0) or w_i h_ik (1 - h_ik)
//                           (which 1); n = pair (e, f), e <= f, B = x_ie x_if
// The tile is GM TM x GN TN outputs, GM GN threads active; rows in steps of BK, the next
// step's h, x and factors in flight (cp.async) while this one is multiplied.
// ------------------------------------------------------------------------------------------
constexpr int OUTER_BK = 16;

template <class T>
struct OuterArgs {
  const T* Xa;
  const T* Ha;
  const T* w;        // OP 1: row weights; OP 0: walpha (N x s)
  int64_t r0, r1;    // rows of the sum
  int64_t rps;       // rows per split
  int d, c, s;
  int which0;        // OP 1: first output kind (0: w h, 1: w h (1 - h))
  int M, Nn;         // outputs in all
  int GM, GN;
  T* part;
};

// FP64: 2 x 2 outputs per thread.
template <int OP>
__global__ __launch_bounds__(512, 1) void k_row_outer_d(const OuterArgs<double> a) {
  constexpr int BK = OUTER_BK, TM = 2, TN = 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int BM = a.GM * TM, BN = a.GN * TN;
  const int d = a.d, c = a.c;
  const int dS = OP == 0 ? BN : (d + 1) & ~1;              // staged x row
  const int bm0 = blockIdx.x * BM, bn0 = blockIdx.y * BN;
  // probes (OP 0) the tile's rows m belong to; one factor per row otherwise
  const int j0 = OP == 0 ? bm0 / c : 0;
  const int nj = OP == 0 ? (min(bm0 + BM, a.M) - 1) / c - j0 + 1 : 1;
  const int njS = OP == 0 ? (BM + c - 1) / c + 1 : 1;
  double* As = (double*)smem_raw;              // [2][BK][BM]
  double* Xs = As + 2 * BK * BM;               // [2][BK][dS]
  double* Ws = Xs + 2 * BK * dS;               // [2][BK][njS]
  double* Bs = Ws + 2 * BK * njS;              // OP 1: [BK][BN]
  int* mcol = (int*)(OP == 0 ? Bs : Bs + BK * BN);   // [BM] class | (probe or kind) << 16
  int* nmap = mcol + BM;                       // OP 1: [BN] e | f << 16
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const int mg = tid / a.GN, ng = tid - mg * a.GN;
  const bool act = mg < a.GM;
  for (int q = tid; q < BM; q += nt) {
    const int m = bm0 + q;
    mcol[q] = m < a.M ? (m % c) | ((OP == 0 ? m / c - j0 : m / c + a.which0) << 16) : -1;
  }
  if (OP == 1)
    for (int q = tid; q < BN; q += nt) {
      int e = 0, f = 0;
      if (bn0 + q < a.Nn) feature_pair(bn0 + q, d, e, f);
      nmap[q] = bn0 + q < a.Nn ? e | (f << 16) : -1;
    }
  __syncthreads();
  const int64_t i0 = a.r0 + (int64_t)blockIdx.z * a.rps;
  const int64_t i1 = min(a.r1, i0 + a.rps);
  const int steps = i0 < i1 ? (int)((i1 - i0 + BK - 1) / BK) : 0;

  auto stage = [&](int t, int b) {
    const int64_t ib = i0 + (int64_t)t * BK;
    double* A = As + b * BK * BM;
    double* X = Xs + b * BK * dS;
    double* W = Ws + b * BK * njS;
    for (int p = wid; p < BK; p += nw) {
      const int64_t i = ib + p;
      const bool rv = i < i1;
      const double* hrow = a.Ha + (rv ? i : a.r0) * c;
      for (int q = lane; q < BM; q += 32) {
        const int mc = mcol[q];
        cp_async<8>(A + p * BM + q, hrow + (mc < 0 ? 0 : mc & 0xffff), rv && mc >= 0);
      }
      const double* xrow = a.Xa + (rv ? i : a.r0) * d;
      const int xo = OP == 0 ? bn0 : 0;
      for (int q = lane; q < dS; q += 32)
        cp_async<8>(X + p * dS + q, xrow + (xo + q < d ? xo + q : 0), rv && xo + q < d);
      if (OP == 0) {
        const double* wrow = a.w + (rv ? i : a.r0) * a.s + j0;
        for (int q = lane; q < nj; q += 32) cp_async<8>(W + p * njS + q, wrow + q, rv);
      } else if (lane == 0) {
        cp_async<8>(W + p, a.w + (rv ? i : a.r0), rv);
      }
    }
    cp_commit();
  };

  double acc[TM][TN] = {};
  if (steps > 0) stage(0, 0);
  for (int t = 0; t < steps; ++t) {
    const int b = t & 1;
    cp_wait0();
    __syncthreads();   // step t has arrived for everyone; step t - 1 is multiplied
    if (t + 1 < steps) stage(t + 1, b ^ 1);
    double* A = As + b * BK * BM;
    const double* X = Xs + b * BK * dS;
    const double* W = Ws + b * BK * njS;
    const int pn = (int)min((int64_t)BK, i1 - i0 - (int64_t)t * BK);
    for (int p = wid; p < pn; p += nw) {
      for (int q = lane; q < BM; q += 32) {
        const int mc = mcol[q] >> 16;
        const double h = A[p * BM + q];
        if (OP == 0) {
          A[p * BM + q] = mc < 0 ? 0.0 : h * W[p * njS + mc];
        } else {
          const double wh = W[p] * h;
          A[p * BM + q] = mc == 1 ? wh * (1.0 - h) : wh;
        }
      }
      if (OP == 1)
        for (int q = lane; q < BN; q += 32) {
          const int ef = nmap[q];
          Bs[p * BN + q] = ef < 0 ? 0.0 : X[p * dS + (ef & 0xffff)] * X[p * dS + (ef >> 16)];
        }
    }
    __syncthreads();
    if (act) {
      const double* B = OP == 0 ? X : Bs;
#pragma unroll 4
      for (int p = 0; p < pn; ++p) {
        const double2 av = *reinterpret_cast<const double2*>(A + p * BM + mg * 2);
        const double2 bv = *reinterpret_cast<const double2*>(B + p * BN + ng * 2);
        acc[0][0] = fma(av.x, bv.x, acc[0][0]);
        acc[0][1] = fma(av.x, bv.y, acc[0][1]);
        acc[1][0] = fma(av.y, bv.x, acc[1][0]);
        acc[1][1] = fma(av.y, bv.y, acc[1][1]);
      }
    }
  }
  if (!act) return;
  double* out = a.part + (int64_t)blockIdx.z * a.M * a.Nn;
#pragma unroll
  for (int x = 0; x < TM; ++x) {
    const int m = bm0 + mg * 2 + x;
    if (m >= a.M) continue;
#pragma unroll
    for (int y = 0; y < TN; ++y) {
      const int n = bn0 + ng * 2 + y;
      if (n < a.Nn) out[(int64_t)m * a.Nn + n] = acc[x][y];
    }
  }
}

// f32, OP 0: 8 x 8 outputs per thread.  Row q of a thread's 8 is tile row
// (q / 4) 4 GM + 4 mg + q % 4, column y is (y / 4) 4 GN + 4 ng + y % 4; a warp covers 8 column
// groups x 4 row groups where GN allows, which is the fewest shared-memory wavefronts.
// One barrier per step.  A step's multiply-adds run in four quarters; each quarter first reads
// its share of the next step's operands (h, its factors and x), multiplies, and then writes that
// share to the other buffer, so that the loads' latency is covered and only one share is held in
// registers.
// Bound by issue slots: the multiply-adds alone run at 53-57 TFLOP/s (78 is the part's peak, 65
// an 8 x 8 outer product from registers), with the operands' loads and stores 40-43 (n = 21,000,
// c = 1000, d = 64, s = 16: 1.08 ms, 2.88 before).  Staging by cp.async with a separate pass over
// the tile ran at 31.
// VH 4: rows of h and x 16-byte aligned, 16 rows per step; otherwise VH values of h per load
// (8-byte aligned rows: 2), x by single values, 8 rows per step.
template <int VH>
struct OuterCfg {
  static constexpr int BK = VH == 4 ? 16 : 8;
  static constexpr int NI = VH == 4 ? 4 : VH == 2 ? 8 : 12;   // loads of h per thread and step
  static constexpr int VX = VH == 4 ? 4 : 1;
  static constexpr int NX = VH == 4 ? 4 : 8;                  // loads of x per thread and step
};
template <int VH>
__global__ __launch_bounds__(256, 2) void k_row_outer_f(const OuterArgs<float> a) {
  using Cfg = OuterCfg<VH>;
  constexpr int BK = Cfg::BK, NI = Cfg::NI, NX = Cfg::NX, VX = Cfg::VX, TM = 8, TN = 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int BM = a.GM * TM, BN = a.GN * TN;
  const int d = a.d, c = a.c;
  const int bm0 = blockIdx.x * BM, bn0 = blockIdx.y * BN;
  const int j0 = bm0 / c;
  float* As = (float*)smem_raw;                // [2][BK][BM]
  float* Bs = As + 2 * BK * BM;                // [2][BK][BN]
  int* mcol = (int*)(Bs + 2 * BK * BN);        // [BM] class | probe << 16
  const int tid = threadIdx.x, nt = blockDim.x;
  int mg, ng;
  if ((a.GN & 7) == 0) {
    mg = (tid >> 3) % a.GM;
    ng = (tid >> 3) / a.GM * 8 + (tid & 7);
  } else {
    mg = tid / a.GN;
    ng = tid - mg * a.GN;
  }
  const bool act = mg < a.GM && ng < a.GN;
  for (int q = tid; q < BM; q += nt) {
    const int m = bm0 + q;
    mcol[q] = m < a.M ? (m % c) | (m / c - j0) << 16 : -1;
  }
  __syncthreads();
  const int64_t i0 = a.r0 + (int64_t)blockIdx.z * a.rps;
  const int64_t i1 = min(a.r1, i0 + a.rps);
  const int rows = i0 < i1 ? (int)(i1 - i0) : 0;
  const int steps = (rows + BK - 1) / BK;
  const int hw = BM / VH, hn = BK * hw;        // loads of h per row and step
  const int xw = BN / VX, xn = BK * xw;        // loads of x
  // the loads' places, fixed over the steps: class | probe << 12 | row of the step << 24
  // (-1: none), and the offset of x
  int hp[NI], xp[NX];
#pragma unroll
  for (int u = 0; u < NI; ++u) {
    const int idx = tid + u * nt, pr = idx / hw, mc = idx < hn ? mcol[(idx - pr * hw) * VH] : -1;
    hp[u] = mc < 0 ? -1 : (mc & 0xffff) | (mc >> 16) << 12 | pr << 24;
  }
#pragma unroll
  for (int u = 0; u < NX; ++u) {
    const int idx = tid + u * nt, pr = idx / xw, q = (idx - pr * xw) * VX;
    xp[u] = idx < xn && bn0 + q < d ? pr * d + q : -1;
  }
  constexpr int QI = NI / 4, QX = NX / 4;   // loads per quarter
  float hr[QI][VH], wr[QI], xr[QX][VX];
  auto load_h = [&](int t, int qt) {
    const int64_t ib = i0 + (int64_t)t * BK;
    const int lim = min(BK, rows - t * BK);
    const float* H = a.Ha + ib * c;
    const float* W = a.w + ib * a.s + j0;
#pragma unroll
    for (int v = 0; v < QI; ++v) {
      const int hu = hp[qt * QI + v], pr = hu >> 24;
#pragma unroll
      for (int z = 0; z < VH; ++z) hr[v][z] = 0.0f;
      wr[v] = 0.0f;
      if (hu >= 0 && pr < lim) {
        const float* h = H + (pr * c + (hu & 0xfff));
        if (VH == 4) {
          const float4 r = *reinterpret_cast<const float4*>(h);
          hr[v][0] = r.x;
          hr[v][VH > 1 ? 1 : 0] = r.y;
          hr[v][VH > 2 ? 2 : 0] = r.z;
          hr[v][VH > 3 ? 3 : 0] = r.w;
        } else if (VH == 2) {
          const float2 r = *reinterpret_cast<const float2*>(h);
          hr[v][0] = r.x;
          hr[v][VH > 1 ? 1 : 0] = r.y;
        } else {
          hr[v][0] = *h;
        }
        wr[v] = W[pr * a.s + (hu >> 12 & 0xfff)];
      }
    }
  };
  auto store_a = [&](int t, int qt) {
    float* A = As + (t & 1) * BK * BM;
#pragma unroll
    for (int v = 0; v < QI; ++v) {
      const int idx = tid + (qt * QI + v) * nt;
      if (idx >= hn) break;
      float r[VH];
#pragma unroll
      for (int z = 0; z < VH; ++z) r[z] = wr[v] * hr[v][z];
      if (VH == 4)
        *reinterpret_cast<float4*>(A + idx * VH) =
            make_float4(r[0], r[VH > 1 ? 1 : 0], r[VH > 2 ? 2 : 0], r[VH > 3 ? 3 : 0]);
      else if (VH == 2)
        *reinterpret_cast<float2*>(A + idx * VH) = make_float2(r[0], r[VH > 1 ? 1 : 0]);
      else
        A[idx] = r[0];
    }
  };
  auto load_x = [&](int t, int qt) {
    const float* X = a.Xa + (i0 + (int64_t)t * BK) * d + bn0;
    const int lim = min(BK, rows - t * BK) * d;   // offsets of a step's rows lie below rows d
#pragma unroll
    for (int v = 0; v < QX; ++v) {
      const int xu = xp[qt * QX + v];
      const bool ok = xu >= 0 && xu < lim;
      if (VX == 4) {
        const float4 r = ok ? *reinterpret_cast<const float4*>(X + xu)
                            : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        xr[v][0] = r.x;
        xr[v][VX > 1 ? 1 : 0] = r.y;
        xr[v][VX > 2 ? 2 : 0] = r.z;
        xr[v][VX > 3 ? 3 : 0] = r.w;
      } else {
        xr[v][0] = ok ? X[xu] : 0.0f;
      }
    }
  };
  auto store_x = [&](int t, int qt) {
    float* X = Bs + (t & 1) * BK * BN;
#pragma unroll
    for (int v = 0; v < QX; ++v) {
      const int idx = tid + (qt * QX + v) * nt;
      if (idx >= xn) break;
      if (VX == 4)
        *reinterpret_cast<float4*>(X + idx * 4) = make_float4(
            xr[v][0], xr[v][VX > 1 ? 1 : 0], xr[v][VX > 2 ? 2 : 0], xr[v][VX > 3 ? 3 : 0]);
      else
        X[idx] = xr[v][0];
    }
  };
  float acc[TM][TN];
#pragma unroll
  for (int x = 0; x < TM; ++x)
#pragma unroll
    for (int y = 0; y < TN; ++y) acc[x][y] = 0.0f;
  if (steps > 0) {
#pragma unroll
    for (int qt = 0; qt < 4; ++qt) {
      load_h(0, qt);
      load_x(0, qt);
      store_a(0, qt);
      store_x(0, qt);
    }
    __syncthreads();
  }
  for (int t = 0; t < steps; ++t) {
    const bool more = t + 1 < steps;
    const float* A = As + (t & 1) * BK * BM + mg * 4;
    const float* B = Bs + (t & 1) * BK * BN + ng * 4;
    const int va = a.GM * 4, vb = a.GN * 4;
#pragma unroll
    for (int qt = 0; qt < 4; ++qt) {
      if (more) {
        load_h(t + 1, qt);
        load_x(t + 1, qt);
      }
      if (act) {
#pragma unroll
        for (int q = 0; q < BK / 4; ++q) {   // rows past the end are zero in both tiles
          float av[TM], bv[TN];
#pragma unroll
          for (int v = 0; v < TM / 4; ++v)
            *reinterpret_cast<float4*>(av + 4 * v) =
                *reinterpret_cast<const float4*>(A + q * BM + v * va);
#pragma unroll
          for (int v = 0; v < TN / 4; ++v)
            *reinterpret_cast<float4*>(bv + 4 * v) =
                *reinterpret_cast<const float4*>(B + q * BN + v * vb);
#pragma unroll
          for (int x = 0; x < TM; ++x)
#pragma unroll
            for (int y = 0; y < TN; ++y) acc[x][y] = fmaf(av[x], bv[y], acc[x][y]);
        }
        A += BK / 4 * BM;
        B += BK / 4 * BN;
      }
      if (more) {
        store_a(t + 1, qt);
        store_x(t + 1, qt);
      }
    }
    __syncthreads();
  }
  if (!act) return;
  float* out = a.part + (int64_t)blockIdx.z * a.M * a.Nn;
#pragma unroll
  for (int x = 0; x < TM; ++x) {
    const int m = bm0 + (x / 4) * a.GM * 4 + mg * 4 + x % 4;
    if (m >= a.M) continue;
#pragma unroll
    for (int y = 0; y < TN; ++y) {
      const int n = bn0 + (y / 4) * a.GN * 4 + ng * 4 + y % 4;
      if (n < a.Nn) out[(int64_t)m * a.Nn + n] = acc[x][y];
    }
  }
}

constexpr size_t OUTER_SMEM = 220 * 1024;   // the most a block of k_row_outer may ask for
template <int OP>
size_t outer_smem_d(int GM, int GN, int d, int c) {
  constexpr int BK = OUTER_BK;
  const int BM = GM * 2, BN = GN * 2;
  const int dS = OP == 0 ? BN : (d + 1) & ~1;
  const int njS = OP == 0 ? (BM + c - 1) / c + 1 : 1;
  size_t el = (size_t)2 * BK * BM + 2 * BK * dS + 2 * BK * njS;
  if (OP == 1) el += (size_t)BK * BN;
  return el * sizeof(double) + ((size_t)BM + (OP == 1 ? BN : 0)) * sizeof(int);
}

bool aligned(const void* q, int bytes) { return reinterpret_cast<uintptr_t>(q) % bytes == 0; }
// values of a row of `cols` f32 that one load may take
int row_vec(const void* q, int cols) {
  return cols % 4 == 0 && aligned(q, 16) ? 4 : cols % 2 == 0 && aligned(q, 8) ? 2 : 1;
}
// k_row_outer_f's VH: 4 needs both operands' rows aligned
int outer_vh(const OuterArgs<float>& a) {
  const int h = row_vec(a.Ha, a.c);
  return h == 4 && row_vec(a.Xa, a.d) == 4 ? 4 : h >= 2 ? 2 : 1;
}
int outer_vh(const OuterArgs<double>&) { return 1; }

// Tile and row splits for M x Nn outputs.
struct OuterPlan {
  int TM, GM, GN, threads, tm, tn, splits;
  int64_t rps;
};

// The tile takes its width from the outputs (groups of TN columns up to 128 of them), then as
// many row groups as the block has threads for (FP64: and shared memory, which one column group
// of up to 512 row groups, d <= 2, exceeds), both cut to equal tiles, so that little of a
// tile is padding at any class count or feature width (the fixed 64 x 64 tile multiplied 54
// empty class columns at c = 10: 413 us a launch at n = 50,000, d = 50, s = 20; now 56).
// Splits: enough blocks for two per SM (one at FP64: 512 threads), whole waves where the row
// count allows it, at most 1024 rows in one f32 sum of the low-rank part, partials of at most
// 512 MiB.  (The block sums take their ranges from block_ranges.)
template <int OP, class T>
OuterPlan outer_plan(const OuterArgs<T>& a, int sms) {
  const bool dbl = sizeof(T) == 8;
  const int M = a.M, Nn = a.Nn, vh = outer_vh(a);
  const int64_t rows = a.r1 - a.r0;
  const int TN = dbl ? 2 : 8;
  OuterPlan p{};
  p.TM = dbl ? 2 : 8;
  const int nt = dbl ? 512 : 256;
  const int max_gn = dbl ? 64 : 16;
  const int ng = (Nn + TN - 1) / TN, mg = (M + p.TM - 1) / p.TM;
  int gn = std::min(ng, max_gn);
  if (mg < nt / gn) gn = std::min(ng, std::min(nt / mg, dbl ? 128 : 64));
  p.tn = (ng + gn - 1) / gn;
  p.GN = (ng + p.tn - 1) / p.tn;
  int gm = std::min(mg, nt / p.GN);
  // f32: the block's threads must also cover a step's loads; FP64: the tile must fit
  const int bk = vh == 4 ? 16 : 8, ni = vh == 4 ? 4 : vh == 2 ? 8 : 12, nx = vh == 4 ? 4 : 8;
  for (;; --gm) {
    p.tm = (mg + gm - 1) / gm;
    p.GM = (mg + p.tm - 1) / p.tm;
    int need = p.GM * p.GN;
    if (!dbl) {
      const int hn = bk * p.GM * p.TM / vh;
      const int xn = bk * p.GN * 8 / (vh == 4 ? 4 : 1);
      need = std::max({need, (hn + ni - 1) / ni, (xn + nx - 1) / nx});
    }
    p.threads = std::max(128, (need + 31) / 32 * 32);
    const bool fits = !dbl || outer_smem_d<OP>(p.GM, p.GN, a.d, a.c) <= OUTER_SMEM;
    if ((p.threads <= nt && fits) || gm == 1) break;
  }
  const int64_t tiles = (int64_t)p.tm * p.tn;
  const int64_t slots = (int64_t)sms * (dbl ? 1 : 2);
  int64_t want = std::max<int64_t>(1, slots / tiles);
  // several waves: round the block count to whole waves
  const int64_t max_rows = dbl ? (int64_t)1 << 40 : 1024;
  want = std::max<int64_t>(want, (rows + max_rows - 1) / max_rows);
  if (want * tiles > slots) {
    const int64_t waves = (want * tiles + slots - 1) / slots;
    want = std::max<int64_t>(want, waves * slots / tiles);
  }
  const int64_t min_rows = dbl ? 4 : 2 * OUTER_BK;
  want = std::min<int64_t>(want, (rows + min_rows - 1) / min_rows);
  const int64_t cap = ((int64_t)1 << 29) / ((int64_t)M * Nn * sizeof(T));
  want = std::max<int64_t>(1, std::min(want, std::max<int64_t>(1, cap)));
  want = std::min<int64_t>(want, 65535);
  p.rps = std::max<int64_t>(1, (rows + want - 1) / want);
  if (!dbl && p.rps > 4 * OUTER_BK) p.rps = ((p.rps + OUTER_BK - 1) / OUTER_BK) * OUTER_BK;
  p.splits = (int)std::max<int64_t>(1, (rows + p.rps - 1) / p.rps);
  return p;
}

template <int VH>
int32_t outer_launch_f(const OuterArgs<float>& a, const OuterPlan& p, cudaStream_t st) {
  const int BK = OuterCfg<VH>::BK, BM = p.GM * 8, BN = p.GN * 8;
  const size_t smem = ((size_t)2 * BK * (BM + BN) + BM) * 4;
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_row_outer_f<VH>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, OUTER_SMEM));
  count_launch();
  k_row_outer_f<VH><<<dim3(p.tm, p.tn, p.splits), p.threads, smem, st>>>(a);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

template <int OP>
int32_t outer_run(OuterArgs<double> a, const OuterPlan& p, cudaStream_t st) {
  a.GM = p.GM;
  a.GN = p.GN;
  a.rps = p.rps;
  const size_t smem = outer_smem_d<OP>(p.GM, p.GN, a.d, a.c);
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_row_outer_d<OP>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, OUTER_SMEM));
  count_launch();
  k_row_outer_d<OP><<<dim3(p.tm, p.tn, p.splits), p.threads, smem, st>>>(a);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

template <int OP>
int32_t outer_run(OuterArgs<float> a, const OuterPlan& p, cudaStream_t st) {
  static_assert(OP == 0, "the f32 block sums are pair_sums");
  a.GM = p.GM;
  a.GN = p.GN;
  a.rps = p.rps;
  const int vh = outer_vh(a);
  if (vh == 4) return outer_launch_f<4>(a, p, st);
  if (vh == 2) return outer_launch_f<2>(a, p, st);
  return outer_launch_f<1>(a, p, st);
}

// ------------------------------------------------------------------------------------------
// reductions over the splits
// ------------------------------------------------------------------------------------------
// Block sums: the triangle's partials, added over the splits in double (8 threads per value,
// fixed order), expanded to the full symmetric block with lam on the diagonal.
template <class T>
__global__ __launch_bounds__(256) void k_pair_expand(const T* __restrict__ part, int splits,
                                                     int64_t count, int64_t stride, int np,
                                                     int d, double lam,
                                                     double* out_d, T* out_t) {
  __shared__ double red[8][33];
  const int64_t idx = blockIdx.x * (int64_t)32 + threadIdx.x;
  double acc = 0.0;
  if (idx < count) {
#pragma unroll 8
    for (int sp = threadIdx.y; sp < splits; sp += 8) acc += (double)part[sp * stride + idx];
  }
  red[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y != 0 || idx >= count) return;
  for (int g = 1; g < 8; ++g) acc += red[g][threadIdx.x];
  const int k = (int)(idx / np);
  int e, f;
  feature_pair((int)(idx - (int64_t)k * np), d, e, f);
  if (e == f) acc += lam;
  const int64_t o1 = ((int64_t)k * d + e) * d + f, o2 = ((int64_t)k * d + f) * d + e;
  if (out_d) out_d[o1] = out_d[o2] = acc;
  if (out_t) out_t[o1] = out_t[o2] = (T)acc;
}

// out_j[k] = S_k V_j[k] - sum over the splits of part[split][j][k]; optional
// pq[j c + k] = V_j[k] . out_j[k].  Block = class k, JB probes x SG groups x dpad features;
// the groups share one output's splits and the terms of S_k V_j[k], added in a fixed order.
template <class T>
__global__ void k_row_combine(const T* __restrict__ S, const T* __restrict__ V,
                              const T* __restrict__ part, int splits, int d, int c, int s,
                              int64_t D, T* __restrict__ out, double* pq, int JB, int SG) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int dpad = (d + 31) & ~31;
  T* vs = (T*)smem_raw;                  // JB * d
  T* gs = vs + (size_t)JB * d;           // SG * JB * dpad (SG > 1)
  __shared__ double red[32];
  const int k = blockIdx.x;
  const int e = threadIdx.x % dpad, q = threadIdx.x / dpad;
  const int g = q / JB, jj = q - g * JB;
  const int j = blockIdx.y * JB + jj;
  for (int idx = threadIdx.x; idx < JB * d; idx += blockDim.x) {
    const int qj = idx / d, f = idx - qj * d;
    const int jx = blockIdx.y * JB + qj;
    vs[idx] = jx < s ? V[(int64_t)jx * D + (int64_t)k * d + f] : T(0);
  }
  __syncthreads();
  T acc = T(0);
  if (j < s && e < d) {
    const T* Sk = S + (int64_t)k * d * d + e;   // S symmetric: column e as row e
#pragma unroll 4
    for (int f = g; f < d; f += SG) acc = fma(Sk[(int64_t)f * d], vs[jj * d + f], acc);
    T ds = T(0);
    const T* dp = part + (int64_t)j * D + (int64_t)k * d + e;
    const int64_t stride = (int64_t)s * D;
#pragma unroll 8
    for (int sp = g; sp < splits; sp += SG) ds += dp[sp * stride];
    acc -= ds;
  }
  for (int h = SG >> 1; h > 0; h >>= 1) {   // SG is a power of two
    T* slot = gs + (size_t)(jj * dpad + e);
    __syncthreads();
    if (g >= h && g < 2 * h) slot[(size_t)g * JB * dpad] = acc;
    __syncthreads();
    if (g < h) acc += slot[(size_t)(g + h) * JB * dpad];
  }
  const bool own = g == 0 && j < s && e < d;
  if (own) out[(int64_t)j * D + (int64_t)k * d + e] = acc;
  if (pq && g == 0) {   // (whole warps; the others have no share)
    double v = own ? (double)vs[jj * d + e] * (double)acc : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (pq && own && e == 0) {
    double tot = 0.0;
    for (int w = 0; w < dpad / 32; ++w) tot += red[(threadIdx.x >> 5) + w];
    pq[(int64_t)j * c + k] = tot;
  }
}

// ------------------------------------------------------------------------------------------
// k_row_form (f32): 128 rows x 128 columns per tile, K = features.
//   MODE 0  alpha:  columns (probe, class), walpha[i][j] = w_i sum_k h_ik (x_i.V_j[k])
//   MODE 1  quad:   64 columns of A_j and the same 64 of B_j;
//           sum_k h a b - (sum_k h a)(sum_k h b) per probe, summed over the block's probes
//   MODE 3  class pairs (Exact-FIRAL): unit (k, l), columns M_kl[e]; sum_e x_e (x.M_kl[e]) times
//           -(2 - delta_kl)(delta_kl h_k - h_k h_l), summed over the block's pairs
//   MODE 2  scores: 64 columns of M1_k and the same 64 of M2_k; q = sum_e x_e (x.M_k[e]),
//           sum over the block's classes of w q1 / (1 + eta w q2), w = h_ik (1 - h_ik)
// The columns of one unit u (probe; class in MODE 2) are its inner index v (class; feature in
// MODE 2) padded to kc, a multiple of 4 not above the tile, and PJ units share a tile when kc
// is small; CC chunks cover inner ranges beyond the tile.  Each thread owns 8 rows and two
// groups of 4 inner indices of one unit, so its share of a row's sum stays in registers; the
// groups meet in shared memory once per tile.  Blocks: 128 rows x a range of units
// (blockIdx.y).
// MODE 2 adds x_e (x.M_k[e]) over the features as sums of two floats (two_prod, two_sum), which
// hold what an FP64 sum does: eq. 14 compares points whose scores differ by little, and f32 sums
// moved them by 1e-8 to 9e-8.  Some 10 f32 instructions a term: a pick takes 620 us at n = 5,000,
// d = c = 50 (605 with f32 sums), 640 at n = 100,000, d = 16, c = 64 (551).  An FP64 multiply-add and
// the conversions of its factors would take the FP64 pipe three times as long as the row's products.
// Bound by issue slots and, per tile, the latency of the row coefficients: 40 TFLOP/s for alpha
// at n = 21,000, c = 1000, d = 64, s = 16 (1.08 ms; one thread per row took 4.67), the quadratic
// forms at n = 50,000, d = 50, c = 10, s = 20 100 us (175 before), the eq. 14 scores at
// n = 5,000, d = c = 50 about 125 us (2,840 before: 40 blocks, one after another over the classes).
// The coefficient tiles are packed first (k_form_pack), feature-major, so that a step of the
// main loop is staged by whole 16-byte copies at any alignment.
// ------------------------------------------------------------------------------------------
constexpr int FORM_LD = 132;    // tile row in shared memory (16-byte rows, no 2-power stride)

struct FormArgs {
  const float* Xa;
  const float* Ha;
  const float* w;        // MODE 0: row weights
  const float* A;        // coefficient blocks, unit u at A + u ustride + v d
  const float* B;        // MODE 1, 2: the second block
  float* pk;             // packed tiles [block y][chunk][tile][dK][128]
  int64_t row0, N;       // first row, end row
  int d, c;
  int units, inner;      // units and inner extent (s, c; MODE 2: c, d)
  int64_t ustride;       // elements between units
  int kc, PJ, CC, UB;    // padded inner chunk, units per tile, chunks, units per block
  int vec;               // float4 reads of the row coefficients are aligned
  double eta;
  const int2* pairs;     // MODE 3
  int64_t ldm;           // MODE 3: row length of M
  float* walpha;         // MODE 0: N x units
  double* part;          // MODE 1, 2: [blockIdx.y][row - row0]
};

// features padded to whole steps of 16
__host__ __device__ inline int form_dk(int d) { return (d + 15) / 16 * 16; }

// hi + lo += b, exactly but for the rounding of lo (two-sum: Knuth, The Art of Computer Programming
// 2, 4.2.2)
__device__ __forceinline__ void two_sum(float& hi, float& lo, float b) {
  const float s = __fadd_rn(hi, b), t = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(b, t)));
  hi = s;
}
// hi + lo += x y: the product's rounding error by one fused multiply-add
__device__ __forceinline__ void two_prod(float& hi, float& lo, float x, float y) {
  const float p = __fmul_rn(x, y);
  lo = __fadd_rn(lo, __fmaf_rn(x, y, -p));
  two_sum(hi, lo, p);
}

// One thread: one tile column, 8 features.
template <int MODE>
__global__ __launch_bounds__(256) void k_form_pack(const FormArgs a, int64_t total) {
  const int dK = form_dk(a.d), eb = dK / 8;
  const int tpb = a.UB / a.PJ;
  for (int64_t idx = blockIdx.x * (int64_t)256 + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * 256) {
    const int col = (int)(idx & 127);
    const int64_t q0 = idx >> 7;
    const int T = (int)(q0 / eb), e0 = (int)(q0 - (int64_t)T * eb) * 8;
    const int p = T % tpb, yc = T / tpb, cc = yc % a.CC, y = yc / a.CC;
    const int q = MODE == 0 || MODE == 3 ? col : col & 63;
    const int ul = q / a.kc, v = cc * a.kc + q - ul * a.kc;
    const int u = y * a.UB + p * a.PJ + ul;
    const bool ok = ul < a.PJ && u < a.units && v < a.inner;
    const float* src = a.A;
    if (MODE == 3) {
      const int2 kl = a.pairs[ok ? u : 0];
      src += ok ? (int64_t)(kl.x * a.d + v) * a.ldm + (int64_t)kl.y * a.d : 0;
    } else {
      if (MODE != 0 && col >= 64) src = a.B;
      src += ok ? u * a.ustride + (MODE == 2 ? v : (int64_t)v * a.d) : 0;
    }
    // MODE 2 takes column v of M_k (symmetric but for the rounding of its f32 products), in runs of
    // consecutive threads
    const int es = MODE == 2 ? a.d : 1;
    float* dst = a.pk + ((int64_t)T * dK + e0) * 128 + col;
#pragma unroll
    for (int e = 0; e < 8; ++e) dst[e * 128] = ok && e0 + e < a.d ? src[(e0 + e) * es] : 0.0f;
  }
}

__host__ __device__ constexpr int form_nv(int mode) {
  return mode == 0 || mode == 3 ? 1 : mode == 1 ? 3 : 2;
}
__host__ __device__ constexpr int form_ns(int mode) { return mode == 2 ? 4 : form_nv(mode); }

// KC features per step: 16, or 8 where that lets two blocks share an SM
template <int MODE, int KC>
__global__ __launch_bounds__(256, 2) void k_row_form(const FormArgs a) {
  constexpr bool ONE = MODE == 0 || MODE == 3;            // one coefficient block
  // values per (row, unit): in red, and in sum as floats (MODE 2: one form at a time as two floats,
  // two forms as doubles)
  constexpr int NV = form_nv(MODE), NS = form_ns(MODE);
  constexpr int GC = ONE ? 32 : 16;                       // column groups per tile
  constexpr int LD = FORM_LD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int d = a.d, dK = form_dk(d);
  float* xs = (float*)smem_raw;              // [dK][LD]
  float* vs = xs + (size_t)dK * LD;          // [2][KC][128]
  float* red = vs + 2 * KC * 128;            // [NV][128][GC + 1]
  float* sum = red + NV * 128 * (GC + 1);    // [NV][UB][128] (MODE 2: doubles, [2][UB][128])
  double* dsum = reinterpret_cast<double*>(sum);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // a warp covers 8 column groups x 4 row groups
  const int tx = (wid & 1) * 8 + (lane & 7), ty = (wid >> 1) * 4 + (lane >> 3);
  const int64_t i0 = a.row0 + (int64_t)blockIdx.x * 128;
  const int u0 = blockIdx.y * a.UB, u1 = min(a.units, u0 + a.UB);
  const int tpb = a.UB / a.PJ;
  const int tpc = (u1 - u0 + a.PJ - 1) / a.PJ;            // tiles per chunk
  const int ntile = a.CC * tpc, nk = dK / KC;
  const int gpu = a.kc / 4;                               // groups per unit
  // x tile, feature-major: 8 features x 4 rows per warp instruction (32-byte reads, no bank
  // conflicts at LD = 132)
  {
    const int el = lane & 7, rl = lane >> 3;
    for (int q = wid; q < 32 * (dK / 8); q += 8) {
      const int r = (q & 31) * 4 + rl, e = (q >> 5) * 8 + el;
      const bool ok = i0 + r < a.N && e < d;
      cp_async<4>(xs + e * LD + r, a.Xa + (ok ? (i0 + r) * d + e : 0), ok);
    }
  }
  for (int q = tid; q < NS * a.UB * 128; q += 256) sum[q] = 0.0f;
  // step kk of tile (cc, p): KC rows of 512 bytes
  auto stage = [&](int cc, int p, int kk, int b) {
    const float* src = a.pk + ((((int64_t)blockIdx.y * a.CC + cc) * tpb + p) * dK + kk * KC) * 128;
    float* dst = vs + b * KC * 128;
#pragma unroll
    for (int x = 0; x < KC / 8; ++x)
      cp_async<16>(dst + (x * 256 + tid) * 4, src + (x * 256 + tid) * 4, true);
    cp_commit();
  };
  stage(0, 0, 0, 0);
  float acc[8][8];
  int step = 0, cc = 0, p = 0;
  for (int t = 0; t < ntile; ++t) {
    const int pn = p + 1 < tpc ? p + 1 : 0, cn = pn ? cc : cc + 1;   // the next tile
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) acc[x][y] = 0.0f;
    for (int kk = 0; kk < nk; ++kk, ++step) {
      const int b = step & 1;
      cp_wait0();
      __syncthreads();
      if (kk + 1 < nk) stage(cc, p, kk + 1, b ^ 1);
      else if (t + 1 < ntile) stage(cn, pn, 0, b ^ 1);
      const float* X = xs + kk * KC * LD + ty * 4;
      const float* Vt = vs + b * KC * 128 + tx * 4;
      // the last step stops at the last feature (the padding is zero)
      const int qn = min(KC, d - kk * KC);
      auto multiply = [&](int q) {
        float av[8], bv[8];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          *reinterpret_cast<float4*>(av + 4 * v) =
              *reinterpret_cast<const float4*>(X + q * LD + v * 64);
          *reinterpret_cast<float4*>(bv + 4 * v) =
              *reinterpret_cast<const float4*>(Vt + q * 128 + v * 64);
        }
#pragma unroll
        for (int x = 0; x < 8; ++x)
#pragma unroll
          for (int y = 0; y < 8; ++y) acc[x][y] = fmaf(av[x], bv[y], acc[x][y]);
      };
      if (qn == KC) {
#pragma unroll 4
        for (int q = 0; q < KC; ++q) multiply(q);
      } else {
        for (int q = 0; q < qn; ++q) multiply(q);
      }
    }
    if (MODE == 2) {
      // the two forms one after the other through the same shared sums
      const int ul = tx / gpu, v = cc * a.kc + (tx - ul * gpu) * 4;
      const bool uv = ul < a.PJ && u0 + p * a.PJ + ul < u1;
      float fh[2][8], fl[2][8];
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const int r = (x / 4) * 64 + ty * 4 + (x & 3);
        fh[0][x] = fl[0][x] = fh[1][x] = fl[1][x] = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float xe = uv && v + q < a.inner ? xs[(v + q) * LD + r] : 0.0f;
          two_prod(fh[0][x], fl[0][x], xe, acc[x][q]);
          two_prod(fh[1][x], fl[1][x], xe, acc[x][4 + q]);
        }
      }
#pragma unroll
      for (int which = 0; which < 2; ++which) {
        if (which) __syncthreads();   // the first form's groups have been added
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          const int r = (x / 4) * 64 + ty * 4 + (x & 3);
          red[r * (GC + 1) + tx] = fh[which][x];
          red[(128 + r) * (GC + 1) + tx] = fl[which][x];
        }
        __syncthreads();
        for (int q = tid; q < a.PJ * 128; q += 256) {
          const int r = q & 127, slot = p * a.PJ + (q >> 7);
          if (u0 + slot < u1) {
            const float* rp = red + r * (GC + 1) + (q >> 7) * gpu;
            float hi = 0.0f, lo = 0.0f;
            for (int x = 0; x < gpu; ++x) {
              two_sum(hi, lo, rp[x]);
              lo = __fadd_rn(lo, rp[128 * (GC + 1) + x]);
            }
            // (an infinite sum's lo is NaN)
            dsum[(which * a.UB + slot) * 128 + r] +=
                isfinite(hi) ? (double)hi + (double)lo : (double)hi;
          }
        }
      }
      cc = cn;
      p = pn;
      continue;
    }
    // per row: this thread's 4 (MODE 0: 2 x 4) inner indices
#pragma unroll
    for (int g = 0; g < (ONE ? 2 : 1); ++g) {
      const int grp = g * 16 + tx;
      const int ul = grp / gpu, v = cc * a.kc + (grp - ul * gpu) * 4;
      const bool uv = ul < a.PJ && u0 + p * a.PJ + ul < u1;
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const int r = (x / 4) * 64 + ty * 4 + (x & 3);
        const int64_t i = i0 + r;
        float cf[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (MODE == 3) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (uv && v + q < a.inner) cf[q] = xs[(v + q) * LD + r];
        } else if (uv && i < a.N) {
          const float* hp = a.Ha + i * a.c + v;
          if (a.vec) {
            if (v < a.inner) {
              const float4 hv = *reinterpret_cast<const float4*>(hp);
              cf[0] = hv.x;
              cf[1] = hv.y;
              cf[2] = hv.z;
              cf[3] = hv.w;
            }
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (v + q < a.inner) cf[q] = hp[q];
          }
        }
        float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float va = acc[x][g * 4 + q], vb = acc[x][4 + q];
          if (ONE) {
            s0 = fmaf(cf[q], va, s0);
          } else {
            const float ha = cf[q] * va;
            s0 = fmaf(ha, vb, s0);
            s1 += ha;
            s2 = fmaf(cf[q], vb, s2);
          }
        }
        red[r * (GC + 1) + grp] = s0;
        if (NV > 1) red[(128 + r) * (GC + 1) + grp] = s1;
        if (NV > 2) red[(256 + r) * (GC + 1) + grp] = s2;
      }
    }
    __syncthreads();
    // groups of one unit, in order; the next write of red is behind at least one barrier
    for (int q = tid; q < NV * a.PJ * 128; q += 256) {
      const int r = q & 127, ul = (q >> 7) % a.PJ, nv = (q >> 7) / a.PJ;
      const int slot = p * a.PJ + ul;
      if (u0 + slot < u1) {
        const float* rp = red + (nv * 128 + r) * (GC + 1) + ul * gpu;
        float acc1 = 0.0f;
        for (int x = 0; x < gpu; ++x) acc1 += rp[x];
        sum[(nv * a.UB + slot) * 128 + r] += acc1;
      }
    }
    cc = cn;
    p = pn;
  }
  __syncthreads();
  if (MODE == 0) {
    for (int q = tid; q < (u1 - u0) * 128; q += 256) {
      const int r = q & 127, ul = q >> 7;
      if (i0 + r < a.N) a.walpha[(i0 + r) * a.units + u0 + ul] = a.w[i0 + r] * sum[ul * 128 + r];
    }
  } else if (tid < 128 && i0 + tid < a.N) {
    const int64_t i = i0 + tid;
    double q = 0.0;
    for (int ul = 0; ul < u1 - u0; ++ul) {
      const double v0 = MODE == 2 ? dsum[ul * 128 + tid] : (double)sum[ul * 128 + tid];
      const double v1 = ONE ? 0.0 : MODE == 2 ? dsum[(a.UB + ul) * 128 + tid]
                                              : (double)sum[(a.UB + ul) * 128 + tid];
      if (MODE == 3) {
        const int2 kl = a.pairs[u0 + ul];
        const double hk = (double)a.Ha[i * a.c + kl.x], hl = (double)a.Ha[i * a.c + kl.y];
        const double w = (kl.x == kl.y ? hk : 0.0) - hk * hl;
        q -= (kl.x == kl.y ? 1.0 : 2.0) * w * v0;
      } else if (MODE == 1) {
        q += v0 - v1 * (double)sum[(2 * a.UB + ul) * 128 + tid];
      } else {
        const double hv = (double)a.Ha[i * a.c + u0 + ul];
        const double wk = hv * (1.0 - hv);
        q += wk * v0 / (1.0 + a.eta * wk * v1);
      }
    }
    a.part[blockIdx.y * (a.N - a.row0) + (i - a.row0)] = q;
  }
}

// Units per tile and block for `rows` rows: kc spreads the inner range over equal chunks of at
// most the tile; units per block: as many as keep the grid's last wave full (two blocks per
// SM), at most `most` (shared-memory sums: 16, or 8 where they are doubles).
void form_plan(FormArgs& a, int tile, int64_t rows, int sms, int most = 16) {
  a.CC = (a.inner + tile - 1) / tile;
  a.kc = ((a.inner + a.CC - 1) / a.CC + 3) / 4 * 4;
  a.PJ = std::min(std::max(1, tile / a.kc), std::min(a.units, most));
  const int64_t rt = (rows + 127) / 128;
  double best = 1e300;
  for (int nb = 1; nb <= most / a.PJ; ++nb) {
    const int ub = nb * a.PJ;
    const int64_t y = (a.units + ub - 1) / ub;
    if (nb > 1 && (nb - 1) * a.PJ >= a.units) break;
    const int64_t waves = (rt * y + 2 * sms - 1) / (2 * sms);
    const double cost = (double)waves * (nb * a.CC + 0.35);   // 0.35: loading the x tile
    if (cost < best) {
      best = cost;
      a.UB = ub;
    }
  }
}

template <int MODE, int KC>
int32_t form_launch_k(const FormArgs& a, int64_t rows, int ny, cudaStream_t st) {
  constexpr int NV = form_nv(MODE), NS = form_ns(MODE);
  constexpr int GC = MODE == 0 || MODE == 3 ? 32 : 16;
  const size_t smem = ((size_t)form_dk(a.d) * FORM_LD + 2 * KC * 128 +
                       (size_t)NV * 128 * (GC + 1) + (size_t)NS * a.UB * 128) *
                      4;
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_row_form<MODE, KC>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  count_launch();
  k_row_form<MODE, KC><<<dim3((unsigned)((rows + 127) / 128), ny), 256, smem, st>>>(a);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

// Per-block row partials (blocks of units x rows x 8 bytes) of at most FORM_PART_BYTES: the rows run
// in chunks of whole tiles beyond that.  Unbounded, Exact-FIRAL's forms would take 10 GB at n = 1 M,
// c = 200, d = 50.  Rows of a chunk:
constexpr int64_t FORM_PART_BYTES = (int64_t)1 << 28;
int64_t form_chunk(int64_t rows, int64_t ny, int tile) {
  const int64_t most = std::max<int64_t>(tile, FORM_PART_BYTES / (8 * ny) / tile * tile);
  return std::min(rows, most);
}

// pack: the coefficients' tiles are not there yet
template <int MODE>
int32_t form_launch(firal_problem* P, FormArgs a, int64_t rows, int* ny, cudaStream_t st,
                    bool pack = true) {
  *ny = (a.units + a.UB - 1) / a.UB;
  const int dK = form_dk(a.d);
  const int64_t tiles = (int64_t)*ny * a.CC * (a.UB / a.PJ);
  FIRAL_TRY(P->form_pk.ensure((size_t)tiles * dK * 128 * sizeof(float)));
  a.pk = P->form_pk.as<float>();
  if (pack) {
    const int64_t total = tiles * (dK / 8) * 128;
    count_launch();
    k_form_pack<MODE><<<(unsigned)std::min<int64_t>((total + 255) / 256, 65536), 256, 0, st>>>(a, total);
  }
  if (a.d <= 96) return form_launch_k<MODE, 16>(a, rows, *ny, st);
  return form_launch_k<MODE, 8>(a, rows, *ny, st);
}

// ------------------------------------------------------------------------------------------
// k_row_form_d (FP64): 32 rows per block, one warp per probe, 4 classes at a time; h is read
// class-major so that a warp's 32 rows are one run.  Bound by the FP64 rate (n = 3,000, d = 20,
// c = s = 10: 20 us a launch, 137 with 128 rows per block; 10 us at 1.25 TFLOP/s).
// ------------------------------------------------------------------------------------------
constexpr int FORM_D_STAGE = 512;   // doubles of a probe's coefficients staged at a time, per warp

template <int MODE>
__global__ __launch_bounds__(256) void k_row_form_d(
    const double* __restrict__ Xa, const double* __restrict__ HaT, const double* __restrict__ w,
    const double* __restrict__ A, const double* __restrict__ B, int64_t row0, int64_t row1, int64_t N,
    int d, int c, int s, int64_t D, double* __restrict__ walpha, double* __restrict__ part) {
  constexpr int KC = 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ldx = d | 1;
  double* xs = (double*)smem_raw;               // [32][ldx]
  double* va = xs + 32 * ldx + (size_t)wid * FORM_D_STAGE;                 // this warp's
  double* vb = va + (size_t)nw * FORM_D_STAGE;                             // MODE 1
  __shared__ double red[8][33];
  const int64_t i0 = row0 + (int64_t)blockIdx.x * 32;
  const int64_t i = i0 + lane;
  const bool rv = i < row1;
  const int j = blockIdx.y * nw + wid;
#pragma unroll 8
  for (int r = wid; r < 32; r += nw)
    for (int e = lane; e < d; e += 32) xs[r * ldx + e] = i0 + r < row1 ? Xa[(i0 + r) * d + e] : 0.0;
  __syncthreads();
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  const double* x = xs + lane * ldx;
  const int ks = max(KC, min((c + KC - 1) / KC * KC, FORM_D_STAGE / d / KC * KC));
  if (j < s) {
    for (int kb = 0; kb < c; kb += ks) {
      const int kn = min(ks, c - kb) * d;
      const int64_t o = (int64_t)j * D + (int64_t)kb * d;
      __syncwarp();
#pragma unroll 4
      for (int q = lane; q < FORM_D_STAGE; q += 32) {
        if (q >= ks * d) break;
        va[q] = q < kn ? A[o + q] : 0.0;
        if (MODE == 1) vb[q] = q < kn ? B[o + q] : 0.0;
      }
      __syncwarp();
      for (int k0 = kb; k0 < min(c, kb + ks); k0 += KC) {
        double ga[KC], gb[KC], hv[KC];
        const double* pa = va + (k0 - kb) * d;
        const double* pb = vb + (k0 - kb) * d;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
          ga[q] = gb[q] = 0.0;
          hv[q] = rv && k0 + q < c ? HaT[(int64_t)(k0 + q) * N + i] : 0.0;
        }
        if (k0 + KC <= c) {
#pragma unroll 2
          for (int e = 0; e < d; ++e) {
            const double xe = x[e];
#pragma unroll
            for (int q = 0; q < KC; ++q) {
              ga[q] = fma(xe, pa[q * d + e], ga[q]);
              if (MODE == 1) gb[q] = fma(xe, pb[q * d + e], gb[q]);
            }
          }
        } else {                   // the last classes: no multiply-adds on padding
          const int kr = c - k0;
          for (int e = 0; e < d; ++e) {
            const double xe = x[e];
#pragma unroll
            for (int q = 0; q < KC - 1; ++q)
              if (q < kr) {
                ga[q] = fma(xe, pa[q * d + e], ga[q]);
                if (MODE == 1) gb[q] = fma(xe, pb[q * d + e], gb[q]);
              }
          }
        }
#pragma unroll
        for (int q = 0; q < KC; ++q) {
          if (MODE == 0) {
            s0 = fma(hv[q], ga[q], s0);
          } else {
            const double ha = hv[q] * ga[q];
            s0 = fma(ha, gb[q], s0);
            s1 += ha;
            s2 = fma(hv[q], gb[q], s2);
          }
        }
      }
    }
  }
  if (MODE == 0) {
    if (j < s && rv) walpha[i * s + j] = w[i] * s0;
    return;
  }
  red[wid][lane] = j < s ? s0 - s1 * s2 : 0.0;
  __syncthreads();
  if (wid == 0 && rv) {
    double q = 0.0;
    for (int x2 = 0; x2 < nw; ++x2) q += red[x2][lane];
    part[blockIdx.y * (row1 - row0) + (i - row0)] = q;
  }
}

// Warps (probes) per block: 4 while the grid is small, so that every block loads all four
// sub-partitions and the blocks spread evenly over the SMs (n = 3,000, s = 10: 285 blocks, at
// most two per SM; 190 blocks of 5 warps took 23 us, 475 of 2 warps, on two sub-partitions, 22),
// up to 8 to share the x tile.
int form_d_warps(int64_t rows, int s, int sms) {
  if ((rows + 31) / 32 * ((s + 7) / 8) < 8LL * sms) return std::min(4, s);
  return (s + (s + 7) / 8 - 1) / ((s + 7) / 8);
}

template <int MODE>
int32_t form_d_launch(const double* Xa, const double* HaT, const double* w, const double* A,
                      const double* B, int64_t row0, int64_t row1, int64_t N, int d, int c, int s,
                      int64_t D, double* walpha, double* part, int nw, cudaStream_t st) {
  const size_t smem = ((size_t)32 * (d | 1) + (size_t)(MODE == 1 ? 2 : 1) * nw * FORM_D_STAGE) * 8;
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_row_form_d<MODE>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  count_launch();
  k_row_form_d<MODE><<<dim3((unsigned)((row1 - row0 + 31) / 32), (s + nw - 1) / nw), nw * 32, smem,
                       st>>>(Xa, HaT, w, A, B, row0, row1, N, d, c, s, D, walpha, part);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

// g_i = -(scale / s) sum over the blocks' partials
template <class T>
__global__ void k_form_sum(const double* __restrict__ part, int ny, int64_t n, double f,
                           T* __restrict__ g) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double q = 0.0;
    for (int y = 0; y < ny; ++y) q += part[y * n + i];
    g[i] = (T)(f * q);
  }
}

// eq. 14: the blocks' partial scores added per row, then the masked argmax of each 128 rows
// (lowest index on ties); r0: the pool's index of the first of the n rows
__global__ __launch_bounds__(128) void k_score_argmax(const double* __restrict__ part, int ny,
                                                      int64_t n, int64_t r0,
                                                      const uint8_t* __restrict__ mask,
                                                      double* part_val, int64_t* part_idx) {
  __shared__ double bv[4];
  __shared__ int64_t bi[4];
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  double val = -INFINITY;
  int64_t idx = INT64_MAX;
  if (i < n && !mask[r0 + i]) {
    double q = 0.0;
    for (int y = 0; y < ny; ++y) q += part[y * n + i];
    if (q == q) {
      val = q;
      idx = r0 + i;
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
    for (int w = 1; w < 4; ++w)
      if (bv[w] > val || (bv[w] == val && bi[w] < idx)) {
        val = bv[w];
        idx = bi[w];
      }
    part_val[blockIdx.x] = val;
    part_idx[blockIdx.x] = idx;
  }
}

// Row ranges of the f32 block sums.  The rows' weights span the labelled rows' 1 and the pool's
// b / n, so a long f32 chain drops part of the small terms: at n = 1M, d = 128, c = 100 Round's
// blocks come out 2e-4 low and its nu 6e-4, and an apply over 400,000 rows and 360 classes
// carries 3e-5.  That error is part of the results and finer ranges would move them by as much, so
// the ranges are those the sums have always had: enough for four blocks per SM at one class a block
// (four classes at d <= 64), rows in order within each.  They follow the SM count, so another device
// or a smaller SM budget adds in other ranges.
void block_ranges(OuterPlan& p, int64_t N, int64_t rows, int d, int c, int sms) {
  const int64_t groups = d > 64 ? c : (c + 3) / 4;
  int64_t n = std::max<int64_t>((4 * (int64_t)sms + groups - 1) / groups, (N + 65535) / 65536);
  n = std::max<int64_t>(1, std::min({n, (N + 255) / 256, (int64_t)4096}));
  p.rps = (N + n - 1) / n;
  p.splits = (int)std::max<int64_t>(1, (rows + p.rps - 1) / p.rps);   // ranges that hold rows
}

// ------------------------------------------------------------------------------------------
// Block sums over feature pairs, f32 (eq. 13's S and B_k with M = (kind, class), Exact-FIRAL's dense
// sums with M = class pair): out[m][p] = sum_i A[i][m] Z[i][p], p a pair e <= f of features,
//   Z = x_e x_f;   A = w h_k (kind 0), w h_k (1 - h_k) (kind 1), wsc w (delta_kl h_k - h_k h_l)
// Both operands are written out first (k_outer_terms), a bounded number of rows of every range at a
// time, so that the product is nothing but copies and multiply-adds: 8 x 16 outputs per thread,
// six 16-byte shared loads per 128 multiply-adds.  Forming A and Z tile by tile inside the product
// cost more issue slots than the operands' traffic costs time: 29 TFLOP/s at n = 21,000, c = 1000,
// d = 64 (3.0 ms), now 44 (1.90 ms and 0.09 for the operands); Exact-FIRAL's sums at n = 5,000,
// c = d = 50 1.02 -> 0.36 ms.  Three blocks per SM at the square tile (168 registers, a few spills
// outside the loop): 408 tiles take one wave of 456 slots, not two of 304 (2.43 ms).  Rows of a
// range are added in order.
// ------------------------------------------------------------------------------------------
struct PairSum {
  const float* Xa;
  const float* Ha;
  const float* w;      // row weights; class pairs: may be null (weights 1), all scaled by wsc
  const int2* pairs;   // class pairs, or null: kinds and classes
  int64_t r0, r1;      // rows of the sum
  int64_t rps;         // rows per range
  int splits;          // ranges
  int d, c, which0;    // which0: the first kind
  float wsc;
  int M, Nn, lda, ldz; // outputs, and row lengths of A and Z (multiples of 4, zero-padded)
  int64_t t0, L;       // this pass: rows [t0, t0 + L) of every range
  float* A;
  float* Z;
  float* part;         // splits x M x Nn
};

constexpr int TERM_ROWS = 16;
__global__ __launch_bounds__(256) void k_outer_terms(const PairSum a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* xs = (float*)smem_raw;   // [TERM_ROWS][d]
  __shared__ float ws[TERM_ROWS];
  const int z = blockIdx.y;
  const int64_t l0 = (int64_t)blockIdx.x * TERM_ROWS;        // row of the pass
  const int64_t i0 = a.r0 + z * a.rps + a.t0 + l0;
  const int64_t end = min(a.r1, a.r0 + (z + 1) * a.rps);
  const int nr = (int)max((int64_t)0, min((int64_t)TERM_ROWS, min(a.L - l0, end - i0)));
  if (nr == 0) return;
  for (int q = threadIdx.x; q < nr * a.d; q += blockDim.x) xs[q] = a.Xa[i0 * a.d + q];
  if (threadIdx.x < nr) ws[threadIdx.x] = a.w ? a.w[i0 + threadIdx.x] : 1.0f;
  __syncthreads();
  const int64_t row = z * a.L + l0;
  const float* H = a.Ha + i0 * a.c;
  float* A = a.A + row * a.lda;
  for (int m = threadIdx.x; m < a.lda; m += blockDim.x) {
    if (a.pairs) {
      const int2 kl = m < a.M ? a.pairs[m] : make_int2(0, 0);
      for (int r = 0; r < nr; ++r) {
        const float hk = H[r * a.c + kl.x];
        const float v = (kl.x == kl.y ? hk : 0.0f) - hk * H[r * a.c + kl.y];
        A[(int64_t)r * a.lda + m] = m < a.M ? a.wsc * ws[r] * v : 0.0f;
      }
    } else {
      const int kind = m / a.c + a.which0, k = m % a.c;
      for (int r = 0; r < nr; ++r) {
        const float h = H[r * a.c + k];
        float v = ws[r] * h;
        if (kind) v *= 1.0f - h;
        A[(int64_t)r * a.lda + m] = m < a.M ? v : 0.0f;
      }
    }
  }
  float* Z = a.Z + row * a.ldz;
  for (int p = threadIdx.x; p < a.ldz; p += blockDim.x) {
    int e = 0, f = 0;
    if (p < a.Nn) feature_pair(p, a.d, e, f);
    for (int r = 0; r < nr; ++r)
      Z[(int64_t)r * a.ldz + p] = p < a.Nn ? xs[r * a.d + e] * xs[r * a.d + f] : 0.0f;
  }
}

// GM thread groups of 8 rows m, 128 / GM of 16 columns: 128 x 128, 64 x 256 or 32 x 512 outputs
template <int GM>
struct PairTile {
  static constexpr int BM = 8 * GM, BN = 16 * (128 / GM), BK = 16, ST = 3;
  static constexpr int SMEM = ST * BK * (BM + BN) * 4;
};
template <int GM>
__global__ __launch_bounds__(128, GM == 16 ? 3 : 2) void k_outer_gemm(const PairSum a) {
  using C = PairTile<GM>;
  constexpr int BM = C::BM, BN = C::BN, BK = C::BK, ST = C::ST, GN = 128 / GM;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* As = (float*)smem_raw;     // [ST][BK][BM]
  float* Zs = As + ST * BK * BM;    // [ST][BK][BN]
  const int tid = threadIdx.x, z = blockIdx.z;
  // a warp covers 32 / GW row groups x GW column groups
  constexpr int GW = GN < 8 ? GN : GM == 16 ? 8 : GN < 32 ? GN : 32;
  const int mg = tid / 32 * (32 / GW) % GM + tid % 32 / GW;
  const int ng = (tid / 32 * (32 / GW) / GM) * GW + tid % GW;
  const int bm0 = blockIdx.x * BM, bn0 = blockIdx.y * BN;
  const int64_t left = min(a.r1, a.r0 + (z + 1) * a.rps) - (a.r0 + z * a.rps + a.t0);
  const int n = (int)max((int64_t)0, min(a.L, left));
  if (n == 0 && a.t0 > 0) return;   // the range ended in an earlier pass
  const int steps = (n + BK - 1) / BK;
  const float* A = a.A + (int64_t)z * a.L * a.lda + bm0;
  const float* Z = a.Z + (int64_t)z * a.L * a.ldz + bn0;
  const int am = a.lda - bm0, zn = a.ldz - bn0;   // columns there are
  auto load = [&](int t) {
    if (t < steps) {
      const int lim = n - t * BK;
      float* As_ = As + t % ST * BK * BM;
      float* Zs_ = Zs + t % ST * BK * BN;
      const float* A_ = A + (int64_t)t * BK * a.lda;
      const float* Z_ = Z + (int64_t)t * BK * a.ldz;
#pragma unroll
      for (int u = 0; u < BK * BM / 512; ++u) {
        const int idx = tid + u * 128, r = idx / (BM / 4), q = idx % (BM / 4) * 4;
        const bool ok = r < lim && q < am;
        cp_async<16>(As_ + r * BM + q, ok ? A_ + (int64_t)r * a.lda + q : a.A, ok);
      }
#pragma unroll
      for (int u = 0; u < BK * BN / 512; ++u) {
        const int idx = tid + u * 128, r = idx / (BN / 4), q = idx % (BN / 4) * 4;
        const bool ok = r < lim && q < zn;
        cp_async<16>(Zs_ + r * BN + q, ok ? Z_ + (int64_t)r * a.ldz + q : a.Z, ok);
      }
    }
    cp_commit();
  };
  float acc[8][16];
  float* out = a.part + (int64_t)z * a.M * a.Nn;
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int m = bm0 + (x / 4) * (BM / 2) + mg * 4 + x % 4;
#pragma unroll
    for (int y = 0; y < 16; ++y) {
      const int p = bn0 + (y / 4) * (BN / 4) + ng * 4 + y % 4;
      acc[x][y] = a.t0 > 0 && m < a.M && p < a.Nn ? out[(int64_t)m * a.Nn + p] : 0.0f;
    }
  }
#pragma unroll
  for (int t = 0; t < ST - 1; ++t) load(t);
  for (int t = 0; t < steps; ++t) {
    cp_wait<ST - 2>();
    __syncthreads();   // step t has landed for all; every thread is done with step t - 1
    load(t + ST - 1);
    const float* As_ = As + t % ST * BK * BM + mg * 4;
    const float* Zs_ = Zs + t % ST * BK * BN + ng * 4;
#pragma unroll 4
    for (int r = 0; r < BK; ++r) {   // rows past the end are zero in both
      float av[8], zv[16];
#pragma unroll
      for (int v = 0; v < 2; ++v)
        *reinterpret_cast<float4*>(av + 4 * v) =
            *reinterpret_cast<const float4*>(As_ + r * BM + v * (BM / 2));
#pragma unroll
      for (int v = 0; v < 4; ++v)
        *reinterpret_cast<float4*>(zv + 4 * v) =
            *reinterpret_cast<const float4*>(Zs_ + r * BN + v * (BN / 4));
#pragma unroll
      for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 16; ++y) acc[x][y] = fmaf(av[x], zv[y], acc[x][y]);
    }
  }
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int m = bm0 + (x / 4) * (BM / 2) + mg * 4 + x % 4;
    if (m >= a.M) continue;
#pragma unroll
    for (int y = 0; y < 16; ++y) {
      const int p = bn0 + (y / 4) * (BN / 4) + ng * 4 + y % 4;
      if (p < a.Nn) out[(int64_t)m * a.Nn + p] = acc[x][y];
    }
  }
}

// The tile that covers M x Nn with the fewest outputs
int pair_tile(int M, int Nn, int64_t* tiles) {
  int best = 16;
  int64_t ba = INT64_MAX;
  for (int gm : {16, 8, 4}) {
    const int bm = 8 * gm, bn = 16 * (128 / gm);
    const int64_t t = (int64_t)((M + bm - 1) / bm) * ((Nn + bn - 1) / bn);
    if (t * bm * bn < ba) {
      ba = t * bm * bn;
      best = gm;
      *tiles = t;
    }
  }
  return best;
}

template <int GM>
int32_t outer_gemm(const PairSum& a, cudaStream_t st) {
  using C = PairTile<GM>;
  FIRAL_CUDA_TRY(cudaFuncSetAttribute(k_outer_gemm<GM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      C::SMEM));
  count_launch();
  k_outer_gemm<GM><<<dim3((a.M + C::BM - 1) / C::BM, (a.Nn + C::BN - 1) / C::BN, a.splits), 128,
                     C::SMEM, st>>>(a);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

// a: everything but the operands' buffers and the passes.  The operands take at most TERM_BYTES
// (and at least TERM_ROWS rows of every range).
constexpr int64_t TERM_BYTES = (int64_t)1 << 29;
int32_t pair_sums(firal_problem* P, PairSum a) {
  cudaStream_t st = P->H->stream;
  a.lda = (a.M + 3) & ~3;
  a.ldz = (a.Nn + 3) & ~3;
  const int64_t row = (int64_t)(a.lda + a.ldz) * sizeof(float);
  const int64_t most = std::max<int64_t>(1, std::min(a.rps, a.r1 - a.r0));   // rows of a range
  a.L = std::max<int64_t>(TERM_ROWS, TERM_BYTES / (row * a.splits) / TERM_ROWS * TERM_ROWS);
  a.L = std::min(a.L, (most + TERM_ROWS - 1) / TERM_ROWS * TERM_ROWS);
  FIRAL_TRY(P->terms.ensure((size_t)(a.L * a.splits * row)));
  a.A = P->terms.as<float>();
  a.Z = a.A + a.L * a.splits * a.lda;
  int64_t tiles = 0;
  const int gm = pair_tile(a.M, a.Nn, &tiles);
  const size_t smem = (size_t)TERM_ROWS * a.d * sizeof(float);
  a.t0 = 0;
  do {
    count_launch();
    k_outer_terms<<<dim3((unsigned)((a.L + TERM_ROWS - 1) / TERM_ROWS), a.splits), 256, smem, st>>>(a);
    FIRAL_CUDA_TRY(cudaGetLastError());
    FIRAL_TRY(gm == 16 ? outer_gemm<16>(a, st) : gm == 8 ? outer_gemm<8>(a, st)
                                                          : outer_gemm<4>(a, st));
    a.t0 += a.L;
  } while (a.t0 < most);
  return FIRAL_OK;
}

template <class T>
int32_t syrk_t(firal_problem* P, const T* w, int64_t rows, double lamS, T* outS, double lamP,
               double* outP) {
  cudaStream_t st = P->H->stream;
  const int d = P->d, c = P->c;
  const int nw = (outS ? 1 : 0) + (outP ? 1 : 0);
  if (nw == 0) return FIRAL_OK;
  const int np = d * (d + 1) / 2;
  const int M = nw * c;
  int splits = 1;
  T* part = nullptr;
  ProfScope ps(st, PF_SYRK);
  if constexpr (sizeof(T) == 8) {
    OuterArgs<T> a{};
    a.Xa = P->Xa.as<T>();
    a.Ha = P->Ha.as<T>();
    a.w = w;
    a.r0 = 0;
    a.r1 = rows;
    a.d = d;
    a.c = c;
    a.s = 1;
    a.which0 = outS ? 0 : 1;
    a.M = M;
    a.Nn = np;
    const OuterPlan p = outer_plan<1>(a, P->sms);
    splits = p.splits;
    FIRAL_TRY(P->syrk_part.ensure((size_t)M * np * splits * sizeof(T)));
    part = a.part = P->syrk_part.as<T>();
    FIRAL_TRY(outer_run<1>(a, p, st));
  } else {
    OuterPlan p{};
    block_ranges(p, P->N, rows, d, c, P->sms);
    splits = p.splits;
    FIRAL_TRY(P->syrk_part.ensure((size_t)M * np * splits * sizeof(T)));
    part = P->syrk_part.as<T>();
    PairSum a{};
    a.Xa = P->Xa.as<float>();
    a.Ha = P->Ha.as<float>();
    a.w = w;
    a.r0 = 0;
    a.r1 = rows;
    a.rps = p.rps;
    a.splits = splits;
    a.d = d;
    a.c = c;
    a.which0 = outS ? 0 : 1;
    a.M = M;
    a.Nn = np;
    a.part = part;
    FIRAL_TRY(pair_sums(P, a));
  }
  const int64_t per = (int64_t)M * np, half = (int64_t)c * np;
  const dim3 blk(32, 8);
  const unsigned grid = (unsigned)((half + 31) / 32);
  if (outS) {
    count_launch();
    k_pair_expand<T><<<grid, blk, 0, st>>>(part, splits, half, per, np, d, lamS, nullptr, outS);
  }
  if (outP) {
    count_launch();
    k_pair_expand<T><<<grid, blk, 0, st>>>(part + (outS ? half : 0), splits, half, per, np, d,
                                           lamP, outP, nullptr);
  }
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

// pw[i] = w_i h_ik over the classes (if hasS), then w_i h_ik (1 - h_ik) (if hasP); blockDim.y rows
// a block
__global__ void k_block_weights(const float* __restrict__ Ha, const float* __restrict__ w,
                                int64_t rows, int c, bool hasS, bool hasP, float* __restrict__ pw) {
  const int cc = (hasS ? c : 0) + (hasP ? c : 0);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.y + threadIdx.y; i < rows;
       i += (int64_t)gridDim.x * blockDim.y) {
    const float wi = w[i];
    for (int k = threadIdx.x; k < c; k += blockDim.x) {
      const float h = Ha[i * c + k], wh = wi * h;
      if (hasS) pw[i * cc + k] = wh;
      if (hasP) pw[i * cc + cc - c + k] = wh * (1.0f - h);
    }
  }
}

// Block sums with every addition in a fixed order: each term is (p x_e) x_f with p = w h (1 - h)
// (and w h for S), rows in order within their range, over the full square, as both (e, f) and
// (f, e) are used.  For results that amplify the sums' rounding: Round's nu and scores (B_k
// alone: its Sigma blocks and B(H_o), firal_precond_blocks), and the classifier refit, whose line
// search compares losses at their f32 noise (S and B_k over few rows).  Also for few (kind, class)
// rows (few_outputs), of which pair_sums multiplies at least 32, after writing every pair of features
// out.  It is OP 0's product with m = (kind and class k, feature e): A = x_e p_k, B = x_f.
constexpr int64_t FEW_ROWS = 256;   // one range at any class count

// Up to 8 (kind, class) rows, a quarter of pair_sums' smallest tile, where either the features are wide
// or the rows many: one apply with s = 1, pair_sums and here, at c = 2: d = 128 2,011 and 400 us at
// n = 100,000, 196 and 112 at 5,000; d = 50 455 and 293 at 100,000 but 106 and 116 at 5,000, where the
// ranges of 256 rows are a chain of latencies (c = 5: 107 and 135).  At d = 50 the lines cross near
// 13,000 rows.
bool few_outputs(int outputs, int d, int64_t rows) {
  return outputs <= 8 && (d > 56 || rows >= 16384);
}

// The same sums, class blocks of d <= DP features padded to DP (64 or 128), one class to DP DP / 128
// threads of 8 x 16 outputs each.  One staged row of x serves both operands: the left one,
// p_k x_e, is formed in registers (8 multiplies to 128 multiply-adds), so staging is nothing but
// asynchronous copies, and a row takes six 16-byte shared loads for 128 multiply-adds (OP 0's 8 x 8
// tile: four for 64, and both operands pass through registers on their way to shared memory).
// Bound by the f32 pipe.  1 M rows, 100 classes, d = 128 (3.3 TFLOP): 75 ms by OP 0, 66 ms here (50 TF/s).
template <int DP, int V>
__global__ __launch_bounds__(128, 2) void k_block_ord(const float* __restrict__ Xa,
                                                      const float* __restrict__ pw, int64_t rows,
                                                      int64_t rps, int d, int cc,
                                                      float* __restrict__ part) {
  constexpr int BK = 16, ST = 4;
  constexpr int TPC = DP * DP / 128, CL = 128 / TPC;   // threads per class, classes per block
  constexpr int NG = DP / 16, NX = BK * DP / V / 128;
  __shared__ __align__(16) float xs[ST][BK][DP];
  __shared__ float ps[ST][BK][CL];
  const int tid = threadIdx.x;
  const int kl = tid / TPC, mg = (tid % TPC) / NG, ng = tid % NG;
  const int k0 = blockIdx.x * CL;
  const int64_t i0 = (int64_t)blockIdx.y * rps, i1 = min(rows, i0 + rps);
  const int n = i0 < i1 ? (int)(i1 - i0) : 0;
  const int steps = (n + BK - 1) / BK;
  auto load = [&](int t) {
    if (t < steps) {
      const int lim = n - t * BK;   // rows left
      const float* X = Xa + (i0 + (int64_t)t * BK) * d;
      float* dst = &xs[t % ST][0][0];
#pragma unroll
      for (int u = 0; u < NX; ++u) {
        const int idx = tid + u * 128, r = idx / (DP / V), q = (idx % (DP / V)) * V;
        const bool ok = r < lim && q < d;
        cp_async<4 * V>(dst + r * DP + q, ok ? X + (int64_t)r * d + q : Xa, ok);
      }
      if (tid < BK * CL) {
        const int r = tid / CL, k = k0 + tid % CL;
        const bool ok = r < lim && k < cc;
        cp_async<4>(&ps[t % ST][r][tid % CL],
                    ok ? pw + (i0 + (int64_t)t * BK + r) * cc + k : pw, ok);
      }
    }
    cp_commit();
  };
  float acc[8][16];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 16; ++y) acc[x][y] = 0.0f;
#pragma unroll
  for (int t = 0; t < ST - 1; ++t) load(t);
  for (int t = 0; t < steps; ++t) {
    cp_wait<ST - 2>();
    __syncthreads();   // step t has landed for all; every thread is done with step t - 1
    load(t + ST - 1);
    const float* X = &xs[t % ST][0][0];
    const float* Pk = &ps[t % ST][0][kl];
#pragma unroll 4
    for (int r = 0; r < BK; ++r) {   // rows past the end: x and p are zero
      float a[8], b[16];
      const float p = Pk[r * CL];
#pragma unroll
      for (int v = 0; v < 2; ++v)
        *reinterpret_cast<float4*>(a + 4 * v) =
            *reinterpret_cast<const float4*>(X + r * DP + v * (DP / 2) + mg * 4);
#pragma unroll
      for (int v = 0; v < 4; ++v)
        *reinterpret_cast<float4*>(b + 4 * v) =
            *reinterpret_cast<const float4*>(X + r * DP + v * (DP / 4) + ng * 4);
#pragma unroll
      for (int x = 0; x < 8; ++x) a[x] *= p;
#pragma unroll
      for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 16; ++y) acc[x][y] = fmaf(a[x], b[y], acc[x][y]);
    }
  }
  if (k0 + kl >= cc) return;
  float* out = part + ((int64_t)blockIdx.y * cc + k0 + kl) * d * d;
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int e = (x / 4) * (DP / 2) + mg * 4 + x % 4;
    if (e >= d) continue;
#pragma unroll
    for (int y = 0; y < 16; ++y) {
      const int f = (y / 4) * (DP / 4) + ng * 4 + y % 4;
      if (f < d) out[e * d + f] = acc[x][y];
    }
  }
}

template <int DP>
int32_t block_ord(const float* Xa, const float* pw, int64_t rows, int64_t rps, int splits, int d,
                  int cc, float* part, cudaStream_t st) {
  constexpr int CL = 128 * 128 / (DP * DP);
  const dim3 grid((unsigned)((cc + CL - 1) / CL), (unsigned)splits);
  count_launch();
  if (row_vec(Xa, d) == 4)
    k_block_ord<DP, 4><<<grid, 128, 0, st>>>(Xa, pw, rows, rps, d, cc, part);
  else
    k_block_ord<DP, 1><<<grid, 128, 0, st>>>(Xa, pw, rows, rps, d, cc, part);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

int32_t blocks_ordered_f32(firal_problem* P, const float* w, int64_t rows, double lamS,
                           float* outS, double lamP, double* outP) {
  cudaStream_t st = P->H->stream;
  const int d = P->d, c = P->c, cc = (outS ? c : 0) + (outP ? c : 0);
  const int64_t per = (int64_t)c * d * d;
  OuterArgs<float> a{};
  a.Xa = a.Ha = P->Xa.as<float>();
  a.r0 = 0;
  a.r1 = rows;
  a.d = a.c = d;
  a.s = cc;
  a.M = cc * d;
  a.Nn = d;
  OuterPlan p = outer_plan<0>(a, P->sms);
  block_ranges(p, P->N, rows, d, c, P->sms);
  FIRAL_TRY(P->syrk_part.ensure((size_t)cc * d * d * p.splits * sizeof(float)));
  FIRAL_TRY(P->blk_w.ensure((size_t)std::max<int64_t>(rows, 1) * cc * sizeof(float)));
  a.part = P->syrk_part.as<float>();
  a.w = P->blk_w.as<float>();
  {
    ProfScope ps(st, PF_SYRK);
    if (rows > 0) {
      count_launch();
      const int tx = std::min(256, (c + 31) / 32 * 32), ty = 256 / tx;
      k_block_weights<<<(unsigned)std::min<int64_t>((rows + ty - 1) / ty, 65536), dim3(tx, ty), 0,
                        st>>>(P->Ha.as<float>(), w, rows, c, outS != nullptr,
                                 outP != nullptr, P->blk_w.as<float>());
      FIRAL_CUDA_TRY(cudaGetLastError());
    }
    // the padded tile where it wastes less than a quarter of its outputs
    if (d > 112)
      FIRAL_TRY(block_ord<128>(a.Xa, a.w, rows, p.rps, p.splits, d, cc, a.part, st));
    else if (d > 56 && d <= 64)
      FIRAL_TRY(block_ord<64>(a.Xa, a.w, rows, p.rps, p.splits, d, cc, a.part, st));
    else
      FIRAL_TRY(outer_run<0>(a, p, st));
  }
  // a range's blocks: S's, then B_k's
  return syrk_reduce_f32(P, a.part, a.part + (outS ? per : 0), p.splits, (int64_t)cc * d * d, lamS,
                         outS, lamP, outP);
}

// The apply of one vector over few rows (the classifier refit's solves), f32, in two launches and
// in a fixed order of additions: alpha row by row (x.V_j[k] by one thread per class, features in
// order; the classes in order by one thread), then per class the rows in order and S_k V_j[k].
__global__ __launch_bounds__(256) void k_few_alpha(const float* __restrict__ Xa,
                                                   const float* __restrict__ Ha,
                                                   const float* __restrict__ w,
                                                   const float* __restrict__ V, int d, int c,
                                                   float* __restrict__ walpha) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* xs = (float*)smem_raw;   // d
  float* gs = xs + d;             // c
  float* hs = gs + c;             // c
  const int64_t i = blockIdx.x;
  for (int e = threadIdx.x; e < d; e += blockDim.x) xs[e] = Xa[i * d + e];
  for (int k = threadIdx.x; k < c; k += blockDim.x) hs[k] = Ha[i * c + k];
  __syncthreads();
  for (int k = threadIdx.x; k < c; k += blockDim.x) {
    const float* v = V + (int64_t)k * d;
    float g = 0.0f;
#pragma unroll 8
    for (int e = 0; e < d; ++e) g = fmaf(xs[e], v[e], g);
    gs[k] = g;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float acc = 0.0f;
#pragma unroll 8
    for (int k = 0; k < c; ++k) acc = fmaf(hs[k], gs[k], acc);
    walpha[i] = w[i] * acc;
  }
}

__global__ __launch_bounds__(128) void k_few_apply(const float* __restrict__ Xa,
                                                   const float* __restrict__ Ha,
                                                   const float* __restrict__ walpha, int rows,
                                                   const float* __restrict__ S,
                                                   const float* __restrict__ V, int d, int c,
                                                   float* __restrict__ out, double* pq) {
  __shared__ float vs[128];
  __shared__ double red[4];
  const int k = blockIdx.x, e = threadIdx.x;
  if (e < d) vs[e] = V[(int64_t)k * d + e];
  __syncthreads();
  float q = 0.0f;
  if (e < d) {
    float ds = 0.0f;
#pragma unroll 8
    for (int i = 0; i < rows; ++i)
      ds = fmaf(walpha[i] * Xa[(int64_t)i * d + e], Ha[(int64_t)i * c + k], ds);
    const float* Sk = S + (int64_t)k * d * d + e;   // S symmetric: column e as row e
    float acc = 0.0f;
#pragma unroll 8
    for (int f = 0; f < d; ++f) acc = fmaf(Sk[(int64_t)f * d], vs[f], acc);
    q = acc - ds;
    out[(int64_t)k * d + e] = q;
  }
  if (!pq) return;
  double v = e < d ? (double)vs[e] * (double)q : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((e & 31) == 0) red[e >> 5] = v;
  __syncthreads();
  if (e == 0) {
    for (int x = 1; x < (int)(blockDim.x >> 5); ++x) v += red[x];
    pq[k] = v;
  }
}

int32_t few_apply(firal_problem* P, const float* w, const float* S, const float* V, float* out,
                  double* pq) {
  cudaStream_t st = P->H->stream;
  const int d = P->d, c = P->c;
  FIRAL_TRY(P->walpha.ensure((size_t)P->N * sizeof(float)));
  {
    ProfScope ps(st, PF_ALPHA);
    count_launch();
    k_few_alpha<<<(unsigned)P->N, std::min(256, (c + 31) / 32 * 32), (d + 2 * c) * sizeof(float),
                  st>>>(P->Xa.as<float>(), P->Ha.as<float>(), w, V, d, c, P->walpha.as<float>());
    FIRAL_CUDA_TRY(cudaGetLastError());
  }
  ProfScope ps(st, PF_DTERM);
  count_launch();
  k_few_apply<<<c, (d + 31) / 32 * 32, 0, st>>>(P->Xa.as<float>(), P->Ha.as<float>(),
                                               P->walpha.as<float>(), (int)P->N, S, V, d, c, out,
                                               pq);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

template <class T>
int32_t apply_t(firal_problem* P, const T* w, const T* Sblk, const T* V, int s, T* out,
                double* pq) {
  cudaStream_t st = P->H->stream;
  const int d = P->d, c = P->c;
  const int64_t N = P->N, D = P->D;
  FIRAL_TRY(P->walpha.ensure((size_t)N * s * sizeof(T)));
  {
    ProfScope ps(st, PF_ALPHA);
    if constexpr (sizeof(T) == 8) {
      FIRAL_TRY(form_d_launch<0>(P->Xa.as<double>(), P->HaT.as<double>(), w, V, nullptr, 0, N, N, d,
                                 c, s, D, P->walpha.as<double>(), nullptr, form_d_warps(N, s, P->sms),
                                 st));
    } else {
      FormArgs a{};
      a.Xa = P->Xa.as<float>();
      a.Ha = P->Ha.as<float>();
      a.w = w;
      a.A = V;
      a.N = N;
      a.d = d;
      a.c = c;
      a.units = s;
      a.inner = c;
      a.ustride = D;
      a.vec = row_vec(a.Ha, c) == 4;
      a.walpha = P->walpha.as<float>();
      form_plan(a, 128, N, P->sms);
      int ny = 0;
      FIRAL_TRY(form_launch<0>(P, a, N, &ny, st));
    }
  }
  OuterArgs<T> o{};
  o.Xa = P->Xa.as<T>();
  o.Ha = P->Ha.as<T>();
  o.w = P->walpha.as<T>();
  o.r0 = 0;
  o.r1 = N;
  o.d = d;
  o.c = c;
  o.s = s;
  o.M = s * c;
  o.Nn = d;
  OuterPlan p = outer_plan<0>(o, P->sms);
  if (forced_splits() > 0) {
    p.splits = (int)std::min<int64_t>(forced_splits(), (N + 31) / 32);
    p.rps = (N + p.splits - 1) / p.splits;
    p.splits = (int)((N + p.rps - 1) / p.rps);
  }
  FIRAL_TRY(P->Dpart.ensure((size_t)p.splits * s * D * sizeof(T)));
  o.part = P->Dpart.as<T>();
  {
    ProfScope ps(st, PF_DTERM);
    FIRAL_TRY(outer_run<0>(o, p, st));
  }
  // the splits over thread groups (a power of two, at most 1024 threads) while the blocks are few,
  // and one probe per block in place of 4 while blocks of 4 would fill less than half the chip
  // (c = 101, d = 100, s = 10: 26 us as 1,010 blocks of one probe, each S_k read ten times; 18 as 303)
  const int dpad = (d + 31) / 32 * 32;
  const int64_t quads = (int64_t)c * ((s + 3) / 4);
  const bool few = quads < 4 * P->sms;
  const int JB = 2 * quads < P->sms ? 1 : 4;
  int SG = 1;
  while (few && 2 * SG * JB * dpad <= 1024 && 2 * SG <= p.splits) SG *= 2;
  const size_t smem = ((size_t)JB * d + (size_t)SG * JB * dpad) * sizeof(T);
  ProfScope ps(st, PF_COMBINE);
  count_launch();
  k_row_combine<T><<<dim3(c, (s + JB - 1) / JB), dpad * JB * SG, smem, st>>>(
      Sblk, V, o.part, p.splits, d, c, s, D, out, pq, JB, SG);
  FIRAL_CUDA_TRY(cudaGetLastError());
  return FIRAL_OK;
}

}  // namespace

int32_t syrk_blocks(firal_problem* P, const void* w, double lamS, void* outS, double lamP,
                    double* outP, int64_t rows) {
  if (rows < 0) rows = P->N;
  const int kinds = (outS ? 1 : 0) + (outP ? 1 : 0);
  if (kinds == 0) return FIRAL_OK;
  if (!P->dbl && (!outS || few_outputs(kinds * P->c, P->d, rows) ||
                  (outP && rows == P->N && rows <= FEW_ROWS)))
    return blocks_ordered_f32(P, (const float*)w, rows, lamS, (float*)outS, lamP, outP);
  if (P->dbl) return syrk_t<double>(P, (const double*)w, rows, lamS, (double*)outS, lamP, outP);
  return syrk_t<float>(P, (const float*)w, rows, lamS, (float*)outS, lamP, outP);
}

int32_t hessian_apply_simt(firal_problem* P, const void* w, const void* Sblk, const void* V,
                           int s, void* out, double* pq) {
  if (P->dbl) {
    FIRAL_TRY(class_major_h(P));
    return apply_t<double>(P, (const double*)w, (const double*)Sblk, (const double*)V, s,
                           (double*)out, pq);
  }
  if (s == 1 && P->N <= FEW_ROWS)
    return few_apply(P, (const float*)w, (const float*)Sblk, (const float*)V, (float*)out, pq);
  return apply_t<float>(P, (const float*)w, (const float*)Sblk, (const float*)V, s, (float*)out,
                        pq);
}

// Per-point quadratic forms (eq. 11): g_i = -(scale/s) sum_j a_j^T H_i b_j for pool rows,
//   a_j^T H_i b_j = sum_k h_ik (x_i.A_j[k]) (x_i.B_j[k]) - (sum_k h_ik x_i.A_j[k])(sum_k h_ik x_i.B_j[k]).
int32_t quad_forms_simt(firal_problem* P, const void* A, const void* B, int s, double scale,
                        void* g) {
  cudaStream_t st = P->H->stream;
  const int d = P->d, c = P->c;
  ProfScope ps(st, PF_QUAD);
  FormArgs a{};
  int nw = 0, ny = 0;
  if (P->dbl) {
    FIRAL_TRY(class_major_h(P));
    nw = form_d_warps(P->n, s, P->sms);
    ny = (s + nw - 1) / nw;
  } else {
    a.Xa = P->Xa.as<float>();
    a.Ha = P->Ha.as<float>();
    a.A = (const float*)A;
    a.B = (const float*)B;
    a.d = d;
    a.c = c;
    a.units = s;
    a.inner = c;
    a.ustride = P->D;
    a.vec = row_vec(a.Ha, c) == 4;
    form_plan(a, 64, P->n, P->sms);
    ny = (s + a.UB - 1) / a.UB;
  }
  const int64_t chunk = form_chunk(P->n, ny, P->dbl ? 32 : 128);
  FIRAL_TRY(P->form_part.ensure((size_t)ny * chunk * sizeof(double)));
  double* part = a.part = P->form_part.as<double>();
  for (int64_t r = 0; r < P->n; r += chunk) {
    const int64_t rows = std::min(chunk, P->n - r);
    const unsigned grid = (unsigned)std::min<int64_t>((rows + 255) / 256, 4096);
    if (P->dbl) {
      FIRAL_TRY(form_d_launch<1>(P->Xa.as<double>(), P->HaT.as<double>(), nullptr,
                                 (const double*)A, (const double*)B, P->m + r, P->m + r + rows,
                                 P->N, d, c, s, P->D, nullptr, part, nw, st));
      count_launch();
      k_form_sum<double><<<grid, 256, 0, st>>>(part, ny, rows, -scale / s, (double*)g + r);
    } else {
      a.row0 = P->m + r;
      a.N = a.row0 + rows;
      FIRAL_TRY(form_launch<1>(P, a, rows, &ny, st, r == 0));
      count_launch();
      k_form_sum<float><<<grid, 256, 0, st>>>(part, ny, rows, -scale / s, (float*)g + r);
    }
    FIRAL_CUDA_TRY(cudaGetLastError());
  }
  return FIRAL_OK;
}

// eq. 14 scores of the pool rows in f32 and the masked argmax of each 128 rows
int32_t round_scores_f32(firal_problem* P, const float* M1, const float* M2, const uint8_t* mask,
                         double eta, double* pv, int64_t* pi, int np) {
  cudaStream_t st = P->H->stream;
  FormArgs a{};
  a.Xa = P->Xa.as<float>();
  a.Ha = P->Ha.as<float>();
  a.A = M1;
  a.B = M2;
  a.d = P->d;
  a.c = P->c;
  a.units = P->c;
  a.inner = P->d;
  a.ustride = (int64_t)P->d * P->d;
  a.eta = eta;
  // sums of 16 classes where two blocks still share an SM
  form_plan(a, 64, P->n, P->sms, P->d <= 80 ? 16 : 8);
  int ny = (a.units + a.UB - 1) / a.UB;
  const int64_t chunk = form_chunk(P->n, ny, 128);
  FIRAL_TRY(P->form_part.ensure((size_t)ny * chunk * sizeof(double)));
  a.part = P->form_part.as<double>();
  ProfScope ps(st, PF_ROUND);
  for (int64_t r = 0; r < P->n; r += chunk) {
    const int64_t rows = std::min(chunk, P->n - r);
    a.row0 = P->m + r;
    a.N = a.row0 + rows;
    FIRAL_TRY(form_launch<2>(P, a, rows, &ny, st, r == 0));
    // (the last chunk's launch also fills the partials past the last row)
    const int64_t blocks = r + rows < P->n ? rows / 128 : np - r / 128;
    count_launch();
    k_score_argmax<<<(unsigned)blocks, 128, 0, st>>>(a.part, ny, rows, r, mask, pv + r / 128,
                                                     pi + r / 128);
    FIRAL_CUDA_TRY(cudaGetLastError());
  }
  return FIRAL_OK;
}

// Exact-FIRAL in f32 (class pairs k <= l).  The partial sums are one product of npairs x d (d +
// 1) / 2 outputs, x x^T being symmetric, and the gradient's forms run on k_row_form: at n = 5,000,
// d = c = 50 1,010 and 1,060 us, where a CTA per class pair over full blocks, and per group of
// pairs with M_kl staged pair by pair, took 1,830 and 2,760.
int32_t pair_sums_f32(firal_problem* P, int64_t r0, int64_t rows, const float* w, double wsc,
                      const int2* pairs, int npairs, DBuf& part, int* splits) {
  PairSum a{};
  a.Xa = P->Xa.as<float>();
  a.Ha = P->Ha.as<float>();
  a.w = w ? w - r0 : nullptr;
  a.r0 = r0;
  a.r1 = r0 + rows;
  a.d = P->d;
  a.c = P->c;
  a.pairs = pairs;
  a.wsc = (float)wsc;
  a.M = npairs;
  a.Nn = P->d * (P->d + 1) / 2;
  // ranges: two blocks per SM, whole waves where the row count allows it, at most 1024 rows in one
  // f32 sum, partials of at most 512 MiB
  int64_t tiles = 1;
  pair_tile(a.M, a.Nn, &tiles);
  const int64_t slots = 2LL * P->sms;
  int64_t want = std::max<int64_t>({1, slots / tiles, (rows + 1023) / 1024});
  if (want * tiles > slots) want = std::max(want, (want * tiles + slots - 1) / slots * slots / tiles);
  want = std::min(want, (rows + 31) / 32);
  want = std::min(want, ((int64_t)1 << 29) / ((int64_t)a.M * a.Nn * 4));
  want = std::max<int64_t>(1, std::min<int64_t>(want, 65535));
  a.rps = std::max<int64_t>(1, (rows + want - 1) / want);
  a.splits = (int)std::max<int64_t>(1, (rows + a.rps - 1) / a.rps);
  FIRAL_TRY(part.ensure((size_t)a.M * a.Nn * a.splits * sizeof(float)));
  a.part = part.as<float>();
  *splits = a.splits;
  ProfScope ps(P->H->stream, PF_EXACT_BUILD);
  return pair_sums(P, a);
}

int32_t pair_forms_f32(firal_problem* P, const int2* pairs, int npairs, const float* M, float* g,
                       bool* done) {
  cudaStream_t st = P->H->stream;
  FormArgs a{};
  a.Xa = P->Xa.as<float>();
  a.Ha = P->Ha.as<float>();
  a.A = M;
  a.d = P->d;
  a.c = P->c;
  a.units = npairs;
  a.inner = P->d;
  a.pairs = pairs;
  a.ldm = P->D;
  form_plan(a, 128, P->n, P->sms);
  const int64_t ny = (npairs + a.UB - 1) / a.UB;
  *done = false;
  // very many classes of few features: the packed tiles would take several times M's memory
  if (ny > 4096) return FIRAL_OK;
  const int64_t chunk = form_chunk(P->n, ny, 128);
  FIRAL_TRY(P->form_part.ensure((size_t)ny * chunk * sizeof(double)));
  a.part = P->form_part.as<double>();
  ProfScope ps(st, PF_EXACT_QUAD);
  for (int64_t r = 0; r < P->n; r += chunk) {
    const int64_t rows = std::min(chunk, P->n - r);
    a.row0 = P->m + r;
    a.N = a.row0 + rows;
    int y = 0;
    FIRAL_TRY(form_launch<3>(P, a, rows, &y, st, r == 0));
    count_launch();
    k_form_sum<float><<<(unsigned)std::min<int64_t>((rows + 255) / 256, 4096), 256, 0, st>>>(
        a.part, y, rows, 1.0, g + r);
    FIRAL_CUDA_TRY(cudaGetLastError());
  }
  *done = true;
  return FIRAL_OK;
}

}  // namespace firal
