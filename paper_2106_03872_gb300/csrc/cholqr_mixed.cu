// Mixed-path CholQR factor (Sec. "Ground-state solution": orthonormalisation of the block by
// the Cholesky factor of its overlap S = Psi^H Psi, Psi <- Psi L^{-H}).
//
// The FP64 factorisation of an n <= 256 matrix in one CTA is bound by GB300's FP64 rate, so
// the factor comes from one FP32 pass refined in FP64:
//
//   1. L1 L1^H = S       FP32 elimination in registers, M1 = L1^{-1}  (one CTA, a cluster from n = 129)
//   2. S2 = M1 S M1^H    FP64 triangular products, S2 = I + E with |E| ~ eps_32 kappa(S)
//   3. M = conj((I - Phi(E)) M1), Phi(E) = strictly lower part of E plus half its diagonal
//
// (I + Phi(E)) is the Cholesky factor of I + E to first order, so (I - Phi(E)) M1 is the
// inverse Cholesky factor of S up to O(E^2) ~ (eps_32 kappa(S))^2 -- below the 24-bit
// precision of the states for kappa(S) up to ~1e4.  A pivot <= tol * S_jj sets status = j + 1
// and M = I.
//
// Without refinement the result is M1 itself (conjugated), accurate to ~eps_32 kappa(S)
// sqrt(n).  The pipelined block iteration takes that form: it uses only the FP32 copy of M,
// whose rounding is of the order of the refinement's correction for the well-conditioned S of
// an iterate, and the next iteration's CholQR starts again from the S of the new block.
#include <cooperative_groups.h>

#include <type_traits>

#include "kernels.h"

namespace ks {

namespace {

constexpr int C32_MAXN = 256;

__device__ __forceinline__ float2 c_mul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// X = L^{-1} of S = L L^H by elimination on the rows of [S | I], in place: after step j columns <= j of
// a row i > j hold its part of L_1^{-1} (L_1 unit lower triangular, S = L_1 D L_1^H) and columns > j the
// reduced matrix, so step j is row_i -= (A_ij / d_j) row_j in all columns but j, which becomes
// -A_ij / d_j.  X = D^{-1/2} L_1^{-1}.  A pivot d_j <= tol S_jj sets status = j + 1.
//
// n dependent steps bound it, so a step is one barrier: the matrix is in registers (row i in CTA
// i mod CL, NR rows a warp, a lane's columns lane + 32 q), and the owner of row j + 1 hands it over in
// shared memory as soon as it has updated it (in a cluster, the other CTAs fetch it from there).  The
// blocked factorisation in shared memory that this replaces kept 8 columns of pivots in one warp,
// three barriers a block, then a second sweep for the inverse: 0.21 ms at n = 128 against 0.11 ms.  With
// the FP64 refinement the factor takes 0.07, 0.18 and 0.35 ms at n = 64, 128 and 200 (0.096, 0.28 and
// 0.79 ms before).
template <int CL, int THREADS, int MAXN> struct Chol {
  static constexpr int Q = MAXN / 32, NWARP = THREADS / 32, NR = MAXN / CL / NWARP;
  struct Shared {
    float2 p[2][MAXN];      // row j at [j & 1] (CL > 1: this CTA's rows)
    float2 pc[2][MAXN];     // CL > 1: the fetched row
    float sjj[MAXN], d[MAXN];
  };
  Shared& sh;
  int n, rank, lane, warp, bad = 0;
  float tol;
  float2 A[NR][Q];

  __device__ __forceinline__ int row(int r) const { return (warp + r * NWARP) * CL + rank; }
  __device__ __forceinline__ Chol(Shared& s, int n_, float tol_) : sh(s), n(n_), tol(tol_) {
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    rank = 0;
    if constexpr (CL > 1) rank = (int)cooperative_groups::this_cluster().block_rank();
  }

  // Steps j in column slot Q1.
  template <int Q1> __device__ __forceinline__ void slot_steps() {
    const int j1 = min(32 * Q1 + 32, n);
    for (int j = 32 * Q1; j < j1; ++j) {
      const int b = j & 1;
      float2* src = sh.p[b];
      if constexpr (CL > 1) {
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        if (threadIdx.x < MAXN) sh.pc[b][threadIdx.x] = cl.map_shared_rank(&sh.p[0][0], j % CL)[b * MAXN + threadIdx.x];
        src = sh.pc[b];
      }
      __syncthreads();
      float2 p[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) p[q] = src[lane + 32 * q];
      const float d = src[j].x;
      if (!(d > tol * sh.sjj[j]) || !isfinite(d)) {                  // uniform
        bad = j + 1;
        return;
      }
      const float inv = __frcp_rn(d);
      if (threadIdx.x == 0) sh.d[j] = d;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int i = row(r);
        if (i > j) {                                                 // warp-uniform
          const float2 l = make_float2(inv * __shfl_sync(0xffffffffu, A[r][Q1].x, j & 31),
                                       inv * __shfl_sync(0xffffffffu, A[r][Q1].y, j & 31));
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            float2 m = A[r][q];
            m.x = fmaf(-l.x, p[q].x, fmaf(l.y, p[q].y, m.x));
            m.y = fmaf(-l.x, p[q].y, fmaf(-l.y, p[q].x, m.y));
            if (q == Q1 && lane == (j & 31)) m = make_float2(-l.x, -l.y);
            A[r][q] = m;
          }
          if (i == j + 1)
#pragma unroll
            for (int q = 0; q < Q; ++q) sh.p[b ^ 1][lane + 32 * q] = A[r][q];
        }
      }
    }
    if constexpr (Q1 + 1 < Q) {
      if (n > 32 * Q1 + 32) slot_steps<Q1 + 1>();
    }
  }

  __device__ __forceinline__ void run(const double2* __restrict__ S, int conj_out, int* __restrict__ status,
                                      double2* __restrict__ Out, float2* __restrict__ Out32) {
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int i = row(r), j = lane + 32 * q;
        A[r][q] = make_float2(0.f, 0.f);
        if (i < n && j < n) {
          // the lower triangle, mirrored
          const double2 v = S[i >= j ? (size_t)i * n + j : (size_t)j * n + i];
          A[r][q] = make_float2((float)v.x, i == j ? 0.f : (i > j ? (float)v.y : -(float)v.y));
        }
      }
    for (int j = threadIdx.x; j < n; j += THREADS) sh.sjj[j] = (float)S[(size_t)j * n + j].x;
    if (warp == 0 && rank == 0)
#pragma unroll
      for (int q = 0; q < Q; ++q) sh.p[0][lane + 32 * q] = A[0][q];
    slot_steps<0>();
    if constexpr (CL > 1) cooperative_groups::this_cluster().sync();   // no CTA leaves while its rows are read
    __syncthreads();                                                 // d
    const float sgn = conj_out ? -1.f : 1.f;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int i = row(r);
      if (i >= n) continue;
      const float f = bad ? 1.f : 1.f / sqrtf(sh.d[i]);
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int j = lane + 32 * q;
        if (j >= n) continue;
        float2 x = make_float2(0.f, 0.f);
        if (i == j)
          x.x = f;
        else if (j < i && !bad)
          x = make_float2(f * A[r][q].x, f * A[r][q].y);
        Out[(size_t)i * n + j] = make_double2((double)x.x, (double)(sgn * x.y));
        if (Out32) Out32[(size_t)i * n + j] = make_float2(x.x, sgn * x.y);
      }
    }
    if (bad && rank == 0 && threadIdx.x == 0) atomicCAS(status, 0, bad);
  }
};

// Writes X = L^{-1} (lower, zeros above; conj(X) when conj_out) of the Hermitian S (n x n, row-major,
// its lower triangle is read) to Out, and an FP32 copy to Out32 when it is given; the identity when S is
// not positive definite.
template <int CL, int THREADS, int MAXN>
__global__ void __launch_bounds__(THREADS, 1)
    k_chol32_inverse(const double2* __restrict__ S, int n, double tol, int conj_out, int* __restrict__ status,
                     double2* __restrict__ Out, float2* __restrict__ Out32) {
  using C = Chol<CL, THREADS, MAXN>;
  __shared__ typename C::Shared sh;
  C c(sh, n, (float)tol);
  c.run(S, conj_out, status, Out, Out32);
}

template <int CL, int THREADS, int MAXN>
void launch_chol32(const double2* S, int n, double tol, int conj_out, int* status, double2* Out, float2* Out32,
                   cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL);
  cfg.blockDim = dim3(THREADS);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  KS_CUDA(cudaLaunchKernelEx(&cfg, k_chol32_inverse<CL, THREADS, MAXN>, S, n, tol, conj_out, status, Out, Out32));
  KS_CHECK_LAUNCH();
}

// Triangular products on 8 x 8 output tiles (64 threads, one output each), K staged through
// shared memory in chunks of 32 with coalesced loads:
//   MODE 0: C = S M^H             C_ij = sum_{k <= j} S_ik conj(M_jk)          (all tiles, FP64)
//   MODE 1: C = M T (lower part)  C_ij = sum_{k <= i} M_ik T_kj, i >= j          (FP64)
//   MODE 2: C = conj(B - Phi(A - I) B) with A = S2 (lower) and B = M1:
//           C_ij = conj(B_ij - sum_{j <= k <= i} Phi_ik B_kj), Phi_ik = A_ik for k < i and
//           (A_ii - 1)/2 for k = i; i >= j, 0 above; C = I once *status is set.  Phi is
//           O(eps_32 kappa), so FP32 products keep the 24-bit accuracy of the rotation.
// MODE 2 also writes an FP32 copy of C to C32 when it is given.
template <int MODE>
__global__ void __launch_bounds__(64) k_tri_product(const double2* __restrict__ A, const double2* __restrict__ B,
                                                    int n, const int* __restrict__ status, double2* __restrict__ C,
                                                    float2* __restrict__ C32) {
  constexpr int KC = 32;
  const int ty = threadIdx.x >> 3, tx = threadIdx.x & 7;
  const int I = blockIdx.y * 8, J = blockIdx.x * 8;
  const int i = I + ty, j = J + tx;
  if (MODE == 2 && *status != 0) {
    if (i < n && j < n) {
      C[(size_t)i * n + j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
      if (C32) C32[(size_t)i * n + j] = make_float2(i == j ? 1.f : 0.f, 0.f);
    }
    return;
  }
  if (MODE != 0 && J > I) {                                          // strictly upper tile
    if (MODE == 2 && i < n && j < n) {
      C[(size_t)i * n + j] = make_double2(0.0, 0.0);
      if (C32) C32[(size_t)i * n + j] = make_float2(0.f, 0.f);
    }
    return;
  }
  // k range of the tile.  The triangles' zeros are stored (M1 above its diagonal) or set while the
  // operands are staged (Phi), where MODE 2 also rounds them, so the products run without tests: the
  // FP64 pipe (two lanes a clock per SM) takes four instructions per complex product.
  const int k0 = MODE == 2 ? J : 0;
  const int k1 = min(n, MODE == 0 ? J + 8 : I + 8);
  using R = typename std::conditional<MODE == 2, float, double>::type;
  using C2 = cplx<R>;
  __shared__ C2 As[8][KC + 1];
  __shared__ C2 Bs[8][KC + 1];                                       // Bs[j][k]
  R re = 0, im = 0;
  for (int kc = k0; kc < k1; kc += KC) {
    for (int e = threadIdx.x; e < 8 * KC; e += 64) {
      const int r = e / KC, k = kc + e % KC;
      double2 a = make_double2(0.0, 0.0), b = a;
      if (I + r < n && k < k1 && (MODE != 2 || k <= I + r)) a = A[(size_t)(I + r) * n + k];
      if (MODE == 2 && k == I + r) a = make_double2(0.5 * (a.x - 1.0), 0.0);   // Phi_ii = (A_ii - 1) / 2
      As[r][e % KC] = mk<C2>((R)a.x, (R)a.y);
      if (MODE == 0) {
        if (J + r < n && k < k1) b = B[(size_t)(J + r) * n + k];
        Bs[r][e % KC] = mk<C2>((R)b.x, (R)b.y);
      } else {
        const int kk = kc + e / 8, jj = e % 8;                        // B rows k, columns J..J+7
        if (kk < k1 && J + jj < n) b = B[(size_t)kk * n + J + jj];
        Bs[jj][e / 8] = mk<C2>((R)b.x, (R)b.y);
      }
    }
    __syncthreads();
    const int kend = min(KC, k1 - kc);
    for (int kk = 0; kk < kend; ++kk) {
      const C2 a = As[ty][kk], b = Bs[tx][kk];
      if (MODE == 0) {                                               // a conj(b)
        re = fma(a.x, b.x, fma(a.y, b.y, re));
        im = fma(a.y, b.x, fma(-a.x, b.y, im));
      } else {
        re = fma(a.x, b.x, fma(-a.y, b.y, re));
        im = fma(a.x, b.y, fma(a.y, b.x, im));
      }
    }
    __syncthreads();
  }
  if (i >= n || j >= n) return;
  if (MODE == 0) {
    C[(size_t)i * n + j] = make_double2((double)re, (double)im);
  } else if (MODE == 1) {
    if (j <= i) C[(size_t)i * n + j] = make_double2((double)re, (double)im);
  } else {
    double2 c = make_double2(0.0, 0.0);
    if (j <= i) {
      const double2 bij = B[(size_t)i * n + j];
      c = make_double2(bij.x - (double)re, -(bij.y - (double)im));
    }
    C[(size_t)i * n + j] = c;
    if (C32) C32[(size_t)i * n + j] = make_float2((float)c.x, (float)c.y);
  }
}

}  // namespace

// M1, T, S2 (n^2 complex128 each)
size_t cholesky_mixed_workspace(int n) { return (size_t)3 * n * n; }

void cholesky_inverse_mixed(const double2* S, double2* M, int n, double tol, double2* work, int* status,
                            cudaStream_t s, float2* M32, bool refine) {
  if (n > C32_MAXN) fail(KS_ERR_ARG, "cholesky_inverse_mixed: n=%d > %d", n, C32_MAXN);
  double2* M1 = work;
  double2* T = work + (size_t)n * n;
  double2* S2 = work + (size_t)2 * n * n;
  auto factor = [&](int conj_out, double2* out, float2* out32) {
    if (n <= SMALL_SUBSPACE)
      chol32_small(S, n, tol, conj_out, status, out, out32, s);
    else if (n <= 32)
      launch_chol32<1, 256, 32>(S, n, tol, conj_out, status, out, out32, s);
    else if (n <= 64)
      launch_chol32<1, 512, 64>(S, n, tol, conj_out, status, out, out32, s);
    else if (n <= 128)
      launch_chol32<1, 1024, 128>(S, n, tol, conj_out, status, out, out32, s);
    else
      launch_chol32<8, 512, 256>(S, n, tol, conj_out, status, out, out32, s);
  };
  if (!refine) {                                                     // the FP32 factor itself
    factor(1, M, M32);
    return;
  }
  const int nt = (n + 7) / 8;
  const dim3 grid(nt, nt);
  factor(0, M1, nullptr);
  k_tri_product<0><<<grid, 64, 0, s>>>(S, M1, n, status, T, nullptr);
  KS_CHECK_LAUNCH();
  k_tri_product<1><<<grid, 64, 0, s>>>(M1, T, n, status, S2, nullptr);   // S2 = M1 S M1^H (lower)
  KS_CHECK_LAUNCH();
  k_tri_product<2><<<grid, 64, 0, s>>>(S2, M1, n, status, M, M32);
  KS_CHECK_LAUNCH();
}

}  // namespace ks
