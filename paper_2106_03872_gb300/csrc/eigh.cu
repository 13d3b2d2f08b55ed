// Hermitian eigen-decomposition of the Rayleigh-Ritz matrix on the mixed path (n <= 256), FP32:
//
//   1. Householder reduction A = Q T Q^H to a real symmetric tridiagonal T (k_tridiag, tridiag.cuh):
//      the n - 1 dependent reflections, one CTA up to 64 rows, then clusters of 2 and 8 CTAs.
//   2. T is split where an off-diagonal element is negligible.  k_tri_vectors: one warp per
//      eigenvalue; its 32 lanes evaluate the Sturm count at 32 interior points of the bracket (33-way
//      multisection) until it is a few ulps of |T| wide, then the vector by twisted factorisation
//      (backward and forward pivots in two lanes at once, twist index at the smallest |gamma|).
//   3. k_tri_degenerate: inside numerically degenerate clusters, inverse iteration from pseudo-random
//      starts with Gram-Schmidt against the earlier members (rare).
//   4. k_ns_gram / k_ns_update: Newton-Schulz steps Z <- Z (3I - Z^T Z) / 2, which pass through once
//      Z^T Z = I to 2e-6 (close but separated eigenvalues leave twisted-factorisation vectors
//      orthogonal only to ~eps |T| / gap).
//   5. k_back_transform: V = H_0 H_1 ... H_{n-2} Z, one warp per vector, its column in registers, the
//      reflectors staged through shared memory ahead of their use.
//
// The FP32 vectors go to complex128 columns; the caller takes the eigenvalues as FP64 Rayleigh
// quotients of these vectors on the FP64 matrix, then sorts and fixes phases (eigh_mixed).
//
// Everything after the reduction is independent per eigenvalue or per output element, so it is spread
// over the GPU.  With the FP64 quotients and the sort it takes 0.17, 0.30, 0.38 and 0.69 ms at n = 64,
// 96, 128 and 200; in one CTA (a Householder solver to n = 128, cyclic Jacobi above) it took 0.36, 0.57,
// 0.80 and 76 ms, and the one-CTA Rayleigh-Ritz step 0.38 and 0.86 ms at n = 64 and 128 where
// rr_step_mixed takes 0.20 and 0.36 ms beside an idle main stream.
//
// rr_step_mixed runs the Rayleigh-Ritz step of one block iteration the same way on the iteration's
// side stream, FP32 in and out (n <= 128):
//   0. H_sub = conj(M) H_raw M^T from the raw projection H_raw = Psi^H (H Psi) and the
//      lower-triangular orthonormaliser M, two products; its Hermitian part is taken as it is loaded;
//   1-5 as above, without the Newton-Schulz steps (the vectors only span the next iterate, whose
//      CholQR orthonormalises the block, and outside degenerate clusters they are orthogonal to
//      eps |T| / gap <= 6e-3);
//   6. C = Vt M and the steepest-descent step matrix Mcat = [(I + alpha Lambda) C | -alpha C] with rows
//      in ascending order of the FP32 eigenvalues.
// H_sub and the vectors are exported so that ritz_values can form the reported FP64 Rayleigh quotients
// off the iteration's critical path.
#include <algorithm>
#include <utility>

#include "kernels.h"
#include "tridiag.cuh"

namespace ks {

namespace {

constexpr int EC_MAXN = 256;
constexpr int RR_MAXN = 128;
constexpr int EC_Q = EC_MAXN / 32;           // row slots of a lane
constexpr unsigned FULLM = 0xffffffffu;
constexpr int NS_STEPS = 3;
constexpr float NS_TOL = 2e-6f;

__device__ __forceinline__ float2 c_mul(float2 a, float2 b) { return tri_mul(a, b); }
__device__ __forceinline__ float2 c_mulc(float2 a, float2 b) {   // conj(a) b
  return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float warp_add(float v) { return tri_sum(v); }

// The matrix: complex128 Hermitian, or the Hermitian part of a complex64 matrix.
struct Load128 {
  const double2* H;
  int n;
  __device__ __forceinline__ float2 operator()(int i, int j) const {
    const double2 h = H[(size_t)i * n + j];
    return make_float2((float)h.x, (float)h.y);
  }
};
struct LoadPart {
  const float2* H;
  int n;
  __device__ __forceinline__ float2 operator()(int i, int j) const {
    const float2 a = H[(size_t)i * n + j], b = H[(size_t)j * n + i];
    return make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
  }
};

template <int CL, int THREADS, int MAXN, class Load>
__global__ void __launch_bounds__(THREADS, 1) k_tridiag(Load load, int n, Tri T) {
  __shared__ TriShared<CL, MAXN> sh;
  if (blockIdx.x == 0 && threadIdx.x < NS_STEPS) T.nserr[threadIdx.x] = 0;
  Tridiag<CL, THREADS, MAXN> t(sh, T, n);
  t.run(load);
}

template <int CL, int THREADS, int MAXN, class Load>
void launch_tridiag(const Load& load, int n, const Tri& T, cudaStream_t s) {
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
  KS_CUDA(cudaLaunchKernelEx(&cfg, k_tridiag<CL, THREADS, MAXN, Load>, load, n, T));
  KS_CHECK_LAUNCH();
}

template <class Load> void tridiag(const Load& load, int n, const Tri& T, cudaStream_t s) {
  if (n <= 32)
    launch_tridiag<1, 256, 32>(load, n, T, s);
  else if (n <= 64)
    launch_tridiag<1, 512, 64>(load, n, T, s);
  else if (n <= 128)
    launch_tridiag<2, 512, 128>(load, n, T, s);
  else
    launch_tridiag<8, 512, 256>(load, n, T, s);
}

// The splitting of T: an off-diagonal element is dropped where it is negligible beside its
// neighbours.  d, e, e2 (after the cuts) to shared memory, |T| to every thread.
__device__ __forceinline__ float load_tridiagonal(const Tri& T, int n, float* d, float* e, float* e2, float* red) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float di = T.d[i], ei = T.e[i];
    const bool cut = i == n - 1 || fabsf(ei) <= 1e-7f * (fabsf(di) + fabsf(T.d[min(i + 1, n - 1)]) + 1e-30f);
    d[i] = di;
    e[i] = cut ? 0.f : ei;
    e2[i] = cut ? 0.f : ei * ei;
  }
  __syncthreads();
  float tn = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    tn = fmaxf(tn, fabsf(d[i]) + fabsf(e[i]) + (i > 0 ? fabsf(e[i - 1]) : 0.f));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tn = fmaxf(tn, __shfl_xor_sync(FULLM, tn, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = tn;
  __syncthreads();
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tn = fmaxf(tn, red[w]);
  return tn;
}

// [b0, b1]: the unreduced block of T that holds row i (e = 0 after its last row)
__device__ __forceinline__ void block_of(const float* e, int n, int i, int lane, int& b0, int& b1) {
  int lo = 0, hi = n - 1;
  for (int j = lane; j < n; j += 32)
    if (e[j] == 0.f) {
      if (j < i) lo = max(lo, j + 1);
      if (j >= i) hi = min(hi, j);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = max(lo, __shfl_xor_sync(FULLM, lo, o));
    hi = min(hi, __shfl_xor_sync(FULLM, hi, o));
  }
  b0 = lo;
  b1 = hi;
}

constexpr int TV_WARPS = 4;

// Eigenvalue `slot` of T and its vector zt[slot][0..n) (zero outside the block), one warp each.
__global__ void __launch_bounds__(32 * TV_WARPS)
    k_tri_vectors(Tri T, int n, float* __restrict__ lam, float* __restrict__ zt) {
  __shared__ float d[EC_MAXN], e[EC_MAXN], e2[EC_MAXN], red[TV_WARPS];
  __shared__ float dm[TV_WARPS][EC_MAXN], dp[TV_WARPS][EC_MAXN];
  const float tnorm = load_tridiagonal(T, n, d, e, e2, red);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int slot = blockIdx.x * TV_WARPS + warp;
  if (slot >= n) return;                                             // warp-uniform; no barrier follows
  int b0, b1;
  block_of(e, n, slot, lane, b0, b1);
  const int kth = slot - b0;
  float lo = 1e30f, hi = -1e30f;                                     // Gershgorin bounds of the block
  for (int i = b0 + lane; i <= b1; i += 32) {
    const float r = (i > b0 ? fabsf(e[i - 1]) : 0.f) + (i < b1 ? fabsf(e[i]) : 0.f);
    lo = fminf(lo, d[i] - r);
    hi = fmaxf(hi, d[i] + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(FULLM, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(FULLM, hi, o));
  }
  const float pad = 1e-6f * fmaxf(fabsf(lo), fabsf(hi)) + 1e-20f;
  lo -= pad;
  hi += pad;
  const float width = 4.8e-7f * tnorm + 1e-30f;                      // ~4 ulps of |T|
  for (int iter = 0; iter < 16 && hi - lo > width; ++iter) {
    const float x = lo + (hi - lo) * (float)(lane + 1) * (1.f / 33.f);
    // Sturm count: eigenvalues of the block below x
    int c = 0;
    float q = d[b0] - x;
    if (fabsf(q) < 1e-30f) q = -1e-30f;
    c += q < 0.f;
    for (int i = b0 + 1; i <= b1; ++i) {
      q = d[i] - x - __fdividef(e2[i - 1], q);
      if (fabsf(q) < 1e-30f) q = -1e-30f;
      c += q < 0.f;
    }
    // new lo: largest x with count <= kth; new hi: smallest x with count >= kth + 1
    float nlo = c <= kth ? x : -1e30f, nhi = c >= kth + 1 ? x : 1e30f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      nlo = fmaxf(nlo, __shfl_xor_sync(FULLM, nlo, o));
      nhi = fminf(nhi, __shfl_xor_sync(FULLM, nhi, o));
    }
    lo = fmaxf(lo, nlo);
    hi = fminf(hi, nhi);
  }
  const float x = 0.5f * (lo + hi);
  if (lane == 0) lam[slot] = x;
  float* z = zt + (size_t)slot * n;
  if (b0 == b1) {
    for (int i = lane; i < n; i += 32) z[i] = i == slot ? 1.f : 0.f;
    return;
  }
  // twisted factorisation: backward pivots in lane 0, forward pivots in lane 1
  const float tiny = 1e-30f + 1e-13f * tnorm;
  float *Dm = dm[warp], *Dp = dp[warp];
  if (lane == 0) {
    float q = d[b1] - x;
    if (fabsf(q) < tiny) q = tiny;
    Dm[b1] = q;
    for (int i = b1 - 1; i >= b0; --i) {
      q = d[i] - x - __fdividef(e2[i], q);
      if (fabsf(q) < tiny) q = tiny;
      Dm[i] = q;
    }
  } else if (lane == 1) {
    float q = d[b0] - x;
    if (fabsf(q) < tiny) q = tiny;
    Dp[b0] = q;
    for (int i = b0 + 1; i <= b1; ++i) {
      q = d[i] - x - __fdividef(e2[i - 1], q);
      if (fabsf(q) < tiny) q = tiny;
      Dp[i] = q;
    }
  }
  __syncwarp();
  // twist index: argmin |gamma_i|, gamma_i = dp_i + dm_i - (d_i - x), lowest index on ties
  float best = 3.4e38f;
  int r = b1;
  for (int i = b0 + lane; i <= b1; i += 32) {
    const float gm = fabsf(Dp[i] + Dm[i] - (d[i] - x));
    if (gm < best) {
      best = gm;
      r = i;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ob = __shfl_xor_sync(FULLM, best, o);
    const int orr = __shfl_xor_sync(FULLM, r, o);
    if (ob < best || (ob == best && orr < r)) {
      best = ob;
      r = orr;
    }
  }
  // z_r = 1; upwards z_i = -(e_i / dp_i) z_{i+1}, downwards z_i = -(e_{i-1} / dm_i) z_{i-1}
  for (int i = b0 + lane; i <= b1; i += 32) {
    if (i < r) Dp[i] = -__fdividef(e[i], Dp[i]);
    if (i > r) Dm[i] = -__fdividef(e[i - 1], Dm[i]);
  }
  __syncwarp();
  if (lane == 0) {
    float v = 1.f;
    for (int i = r - 1; i >= b0; --i) {
      v *= Dp[i];
      Dp[i] = v;
    }
  } else if (lane == 1) {
    float v = 1.f;
    for (int i = r + 1; i <= b1; ++i) {
      v *= Dm[i];
      Dm[i] = v;
    }
  }
  __syncwarp();
  float nrm = 0.f;
  for (int i = b0 + lane; i <= b1; i += 32) {
    const float v = i < r ? Dp[i] : (i > r ? Dm[i] : 1.f);
    nrm += v * v;
  }
  nrm = warp_add(nrm);
  const float inv = rsqrtf(nrm);
  for (int i = lane; i < n; i += 32) {
    float v = 0.f;
    if (i >= b0 && i <= b1) v = inv * (i < r ? Dp[i] : (i > r ? Dm[i] : 1.f));
    z[i] = v;
  }
}

constexpr int DG_WARPS = 16;

// Degenerate clusters of a block (gaps <= 1e-5 |T|): the twisted factorisation returns nearly the
// same vector for every member, so each member after the first is recomputed by two inverse
// iterations from a pseudo-random start, each followed by Gram-Schmidt against the cluster's
// earlier members (the scheme of LAPACK's stein).  One warp per block of T.
__global__ void __launch_bounds__(32 * DG_WARPS)
    k_tri_degenerate(Tri T, int n, const float* __restrict__ lam, float* __restrict__ zt) {
  __shared__ float d[EC_MAXN], e[EC_MAXN], e2[EC_MAXN], ls[EC_MAXN], red[DG_WARPS];
  __shared__ float Ls[DG_WARPS][EC_MAXN], Ys[DG_WARPS][EC_MAXN];
  const float tnorm = load_tridiagonal(T, n, d, e, e2, red);
  for (int i = threadIdx.x; i < n; i += blockDim.x) ls[i] = lam[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float tiny = 1e-30f + 1e-13f * tnorm;
  float *L = Ls[warp], *Y = Ys[warp];
  for (int b = warp; b < n; b += DG_WARPS) {
    if (b > 0 && e[b - 1] != 0.f) continue;                          // not the first row of a block
    int b0, b1;
    block_of(e, n, b, lane, b0, b1);
    for (int j = b + 1; j <= b1; ++j) {
      int c0 = j;
      while (c0 > b && ls[c0] - ls[c0 - 1] <= 1e-5f * tnorm) --c0;
      if (c0 == j) continue;
      for (int i = b + lane; i <= b1; i += 32) {
        const unsigned hsh = (unsigned)(i * 131 + j * 7919) * 2654435761u;
        Y[i] = (float)(hsh >> 16) * (1.f / 32768.f) - 1.f;
      }
      __syncwarp();
      const float lj = ls[j];
      for (int it = 0; it < 2; ++it) {
        if (lane == 0) {
          float piv = d[b] - lj;
          if (fabsf(piv) < tiny) piv = tiny;
          float u = Y[b];
          Y[b] = __fdividef(u, piv);
          for (int i = b + 1; i <= b1; ++i) {
            const float l = __fdividef(e[i - 1], piv);
            L[i - 1] = l;
            piv = d[i] - lj - l * e[i - 1];
            if (fabsf(piv) < tiny) piv = tiny;
            u = Y[i] - l * u;
            Y[i] = __fdividef(u, piv);
          }
          for (int i = b1 - 1; i >= b; --i) Y[i] -= L[i] * Y[i + 1];
        }
        __syncwarp();
        for (int p = c0; p < j; ++p) {
          const float* zp = zt + (size_t)p * n;
          float sd = 0.f;
          for (int i = b + lane; i <= b1; i += 32) sd += zp[i] * Y[i];
          sd = warp_add(sd);
          for (int i = b + lane; i <= b1; i += 32) Y[i] -= sd * zp[i];
          __syncwarp();
        }
        float sn = 0.f;
        for (int i = b + lane; i <= b1; i += 32) sn += Y[i] * Y[i];
        sn = warp_add(sn);
        const float inv = rsqrtf(fmaxf(sn, 1e-30f));
        for (int i = b + lane; i <= b1; i += 32) Y[i] *= inv;
        __syncwarp();
      }
      for (int i = b + lane; i <= b1; i += 32) zt[(size_t)j * n + i] = Y[i];
      __syncwarp();
    }
  }
}

// One 32 x 32 tile of G = Z^T Z (zt holds the vectors as rows), 256 threads of 2 x 2 outputs, and
// the largest deviation from the identity.
__global__ void __launch_bounds__(256) k_ns_gram(const float* __restrict__ zt, int n, float* __restrict__ G,
                                                 int* __restrict__ err) {
  __shared__ float As[32][33], Bs[32][33];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, a0 = blockIdx.y * 32, b0 = blockIdx.x * 32;
  float g[2][2] = {};
  for (int k0 = 0; k0 < n; k0 += 32) {
    for (int q = threadIdx.x; q < 1024; q += 256) {
      const int r = q >> 5, c = q & 31;
      As[r][c] = (a0 + r < n && k0 + c < n) ? zt[(size_t)(a0 + r) * n + k0 + c] : 0.f;
      Bs[r][c] = (b0 + r < n && k0 + c < n) ? zt[(size_t)(b0 + r) * n + k0 + c] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 32; ++c)
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) g[u][v] += As[ty + 16 * u][c] * Bs[tx + 16 * v][c];
    __syncthreads();
  }
  float dev = 0.f;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int a = a0 + ty + 16 * u, b = b0 + tx + 16 * v;
      if (a < n && b < n) {
        G[(size_t)a * n + b] = g[u][v];
        dev = fmaxf(dev, fabsf(g[u][v] - (a == b ? 1.f : 0.f)));
      }
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dev = fmaxf(dev, __shfl_xor_sync(FULLM, dev, o));
  if ((threadIdx.x & 31) == 0) atomicMax(err, __float_as_int(dev));   // dev >= 0: bits order as the values
}

// out = 1.5 Z - 0.5 Z G, or Z itself where Z^T Z = I already
__global__ void __launch_bounds__(256) k_ns_update(const float* __restrict__ zt, const float* __restrict__ G, int n,
                                                   const int* __restrict__ err, float* __restrict__ out) {
  __shared__ float Gs[32][33], Zs[32][33];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, a0 = blockIdx.y * 32, i0 = blockIdx.x * 32;
  const bool step = __int_as_float(*err) > NS_TOL;                   // uniform over the grid
  float z[2][2] = {};
  if (step)
    for (int k0 = 0; k0 < n; k0 += 32) {
      for (int q = threadIdx.x; q < 1024; q += 256) {
        const int r = q >> 5, c = q & 31;
        Gs[r][c] = (a0 + r < n && k0 + c < n) ? G[(size_t)(a0 + r) * n + k0 + c] : 0.f;   // G symmetric
        Zs[r][c] = (k0 + r < n && i0 + c < n) ? zt[(size_t)(k0 + r) * n + i0 + c] : 0.f;
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 32; ++c)
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int v = 0; v < 2; ++v) z[u][v] += Gs[ty + 16 * u][c] * Zs[c][tx + 16 * v];
      __syncthreads();
    }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int a = a0 + ty + 16 * u, i = i0 + tx + 16 * v;
      if (a < n && i < n) {
        const float c = zt[(size_t)a * n + i];
        out[(size_t)a * n + i] = step ? 1.5f * c - 0.5f * z[u][v] : c;
      }
    }
}

constexpr int BK_WARPS = 4;      // eigenvectors per CTA
constexpr int BK_CH = 8;         // reflectors per staged chunk

// V = H_0 ... H_{n-2} Z, one warp per column; row i = lane + 32 p of the column in slot p.  Out [n][n]
// (column j = vector j) in complex128 or complex64.
template <class Out>
__global__ void __launch_bounds__(32 * BK_WARPS)
    k_back_transform(Tri T, int n, const float* __restrict__ zt, Out* __restrict__ V) {
  __shared__ __align__(16) float2 Rs[2][BK_CH][EC_MAXN];
  __shared__ float2 taus[EC_MAXN];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = blockIdx.x * BK_WARPS + warp;
  const int nr = n - 1, nch = (nr + BK_CH - 1) / BK_CH, ldr = T.ldr;
  for (int k = threadIdx.x; k < nr; k += blockDim.x) taus[k] = T.tau[k];
  // chunk c: reflectors nr - 1 - (c BK_CH + r), the last one first; rows of ldr (a multiple of 32)
  auto stage = [&](int c) {
    for (int q = threadIdx.x; q < BK_CH * (ldr / 2); q += blockDim.x) {
      const int r = q / (ldr / 2), w = q - r * (ldr / 2), k = nr - 1 - (c * BK_CH + r);
      if (k >= 0)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                         (unsigned)__cvta_generic_to_shared(&Rs[c & 1][r][2 * w])),
                     "l"(T.R + (size_t)k * ldr + 2 * w));
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  float2 v[EC_Q];
#pragma unroll
  for (int p = 0; p < EC_Q; ++p) {
    const int i = lane + 32 * p;
    v[p] = make_float2((i < n && j < n) ? zt[(size_t)j * n + i] : 0.f, 0.f);
  }
  if (nch > 0) stage(0);
  for (int c = 0; c < nch; ++c) {
    if (c + 1 < nch) {
      stage(c + 1);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    for (int r = 0; r < BK_CH; ++r) {
      const int k = nr - 1 - (c * BK_CH + r);
      if (k < 0) break;
      const float2 tk = taus[k];
      if (tk.x == 0.f && tk.y == 0.f) continue;                      // uniform
      const int p0 = (k + 1) >> 5;                                   // slots below hold rows <= k only
      float2 rv[EC_Q], dot = make_float2(0.f, 0.f);
#pragma unroll
      for (int p = 0; p < EC_Q; ++p)
        if (p >= p0 && 32 * p < ldr) {
          rv[p] = Rs[c & 1][r][lane + 32 * p];
          const float2 m = c_mulc(rv[p], v[p]);
          dot.x += m.x;
          dot.y += m.y;
        }
      dot.x = warp_add(dot.x);
      dot.y = warp_add(dot.y);
      const float2 f = c_mul(tk, dot);
#pragma unroll
      for (int p = 0; p < EC_Q; ++p)
        if (p >= p0 && 32 * p < ldr) {
          const float2 m = c_mul(rv[p], f);
          v[p].x -= m.x;
          v[p].y -= m.y;
        }
    }
    __syncthreads();                                                 // the chunk's buffer is free
  }
  if (j < n)
#pragma unroll
    for (int p = 0; p < EC_Q; ++p) {
      const int i = lane + 32 * p;
      if (i < n) {
        Out o;
        o.x = v[p].x;
        o.y = v[p].y;
        V[(size_t)i * n + j] = o;
      }
    }
}

// C = opA(A) opB(B) for n x n complex64 matrices, one 32 x 32 tile per CTA (256 threads of 2 x 2
// outputs): FP32 products summed in FP32 over K chunks of 32, the chunks in FP64.
//   MODE 0: A_ik B_jk, k <= j (B lower triangular)                      T = H_raw M^T
//   MODE 1: conj(A_ik) B_kj, k <= i (A lower triangular)                H_sub = conj(M) T
//   MODE 2: A_ki B_kj, k >= j (B lower triangular)                      C = Vt M, then Mcat's rows
struct MatOut {
  float2* C;            // MODE 0, 1: [n][n]
  float2* Mcat;         // MODE 2: [n][2n]
  const float* lam;
  float alpha;
  int* perm;
};
template <int MODE>
__global__ void __launch_bounds__(256) k_rr_product(const float2* __restrict__ A, const float2* __restrict__ B, int n,
                                                    MatOut out) {
  __shared__ float2 As[32][33], Bs[32][33];                          // As[k][i], Bs[k][j]
  __shared__ float ls[RR_MAXN];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  const float2 zero = make_float2(0.f, 0.f);
  double2 sum[2][2] = {};
  const int kb = MODE == 2 ? j0 : 0;                                 // the triangle's range, in whole chunks
  const int ke = MODE == 0 ? min(n, j0 + 32) : (MODE == 1 ? min(n, i0 + 32) : n);
  if (MODE == 2)
    for (int j = threadIdx.x; j < n; j += 256) ls[j] = out.lam[j];
  for (int k0 = kb; k0 < ke; k0 += 32) {
    __syncthreads();
    for (int q = threadIdx.x; q < 1024; q += 256) {
      const int r = q >> 5, c = q & 31;
      if (MODE == 2) {
        As[r][c] = (k0 + r < n && i0 + c < n) ? A[(size_t)(k0 + r) * n + i0 + c] : zero;
      } else {
        As[c][r] = (i0 + r < n && k0 + c < n) ? A[(size_t)(i0 + r) * n + k0 + c] : zero;
      }
      if (MODE == 0)
        Bs[c][r] = (j0 + r < n && k0 + c < n) ? B[(size_t)(j0 + r) * n + k0 + c] : zero;
      else
        Bs[r][c] = (k0 + r < n && j0 + c < n) ? B[(size_t)(k0 + r) * n + j0 + c] : zero;
    }
    __syncthreads();
    float2 acc[2][2] = {};
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      float2 a[2], b[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        a[u] = As[k][ty + 16 * u];
        if (MODE == 1) a[u].y = -a[u].y;
        b[u] = Bs[k][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          acc[u][v].x = fmaf(a[u].x, b[v].x, fmaf(-a[u].y, b[v].y, acc[u][v].x));
          acc[u][v].y = fmaf(a[u].x, b[v].y, fmaf(a[u].y, b[v].x, acc[u][v].y));
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        sum[u][v].x += (double)acc[u][v].x;
        sum[u][v].y += (double)acc[u][v].y;
      }
  }
  if (MODE == 2) __syncthreads();                                    // ls, where the loop ran no chunk
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int i = i0 + ty + 16 * u;
    if (i >= n) continue;
    float f = 0.f;
    float2* row = nullptr;
    if (MODE == 2) {
      // the vector's rank (ties by index) is its row in Mcat
      const float li = ls[i];
      int rank = 0;
      for (int j = 0; j < n; ++j) rank += (ls[j] < li) || (ls[j] == li && j < i);
      f = 1.f + out.alpha * li;
      row = out.Mcat + (size_t)rank * 2 * n;
      if (blockIdx.x == 0 && tx == 0) out.perm[i] = rank;
    }
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int j = j0 + tx + 16 * v;
      if (j >= n) continue;
      const float2 c = make_float2((float)sum[u][v].x, (float)sum[u][v].y);
      if (MODE == 2) {
        row[j] = make_float2(f * c.x, f * c.y);
        row[n + j] = make_float2(-out.alpha * c.x, -out.alpha * c.y);
      } else {
        out.C[(size_t)i * n + j] = c;
      }
    }
  }
}

// Reported eigenvalues of the Rayleigh-Ritz variant: FP64 Rayleigh quotients of the FP32
// eigenvectors on the FP32 subspace matrix (of its Hermitian part, the real part of the quotient),
// eig[perm[j]] = Re(v_j^H A v_j) / (v_j^H v_j).
__global__ void k_ritz_values(const float2* __restrict__ A, const float2* __restrict__ V, const int* __restrict__ perm,
                              int n, double* __restrict__ eig) {
  const int j = blockIdx.x;
  __shared__ double2 v[RR_MAXN];
  __shared__ double red[2][8];
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const float2 x = V[k * n + j];
    v[k] = make_double2((double)x.x, (double)x.y);
  }
  __syncthreads();
  double num = 0.0, den = 0.0;
  for (int a = threadIdx.x >> 5; a < n; a += blockDim.x >> 5) {
    const double2 va = v[a];
    double2 s = make_double2(0.0, 0.0);
    for (int b = threadIdx.x & 31; b < n; b += 32) {
      const float2 h = A[a * n + b];
      const double2 vb = v[b];
      s.x += (double)h.x * vb.x - (double)h.y * vb.y;
      s.y += (double)h.x * vb.y + (double)h.y * vb.x;
    }
    num += va.x * s.x + va.y * s.y;                                  // Re(conj(v_a) s)
    if ((threadIdx.x & 31) == 0) den += va.x * va.x + va.y * va.y;
  }
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(FULLM, num, o);
    den += __shfl_xor_sync(FULLM, den, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = num;
    red[1][threadIdx.x >> 5] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    eig[perm[j]] = a / b;
  }
}

}  // namespace

// One decomposition's small arrays, G and the reflectors, laid out in `work`.
static Tri lay_out(void* work, int n, float*& lam, float*& G) {
  Tri T;
  T.tau = static_cast<float2*>(work);
  T.d = reinterpret_cast<float*>(T.tau + EC_MAXN);
  T.e = T.d + EC_MAXN;
  lam = T.e + EC_MAXN;
  T.nserr = reinterpret_cast<int*>(lam + EC_MAXN);
  G = lam + EC_MAXN + 4;                                             // 16-byte aligned, as the reflectors are
  T.ldr = (n + 31) / 32 * 32;
  T.R = reinterpret_cast<float2*>(G + ((size_t)n * n + 3) / 4 * 4);
  return T;
}

size_t eigh_workspace(int n) {
  const size_t nn = (size_t)n * n;
  return EC_MAXN * (sizeof(float2) + 3 * sizeof(float)) + 4 * sizeof(float) + (nn + 3) / 4 * 4 * sizeof(float) +
         (size_t)n * ((n + 31) / 32 * 32) * sizeof(float2);
}

void eigh_vectors_f32(const double2* A, double2* V, int n, void* work, void* work2, cudaStream_t s) {
  if (n > EC_MAXN || n < 1) fail(KS_ERR_ARG, "eigh_vectors_f32: n=%d not in [1, %d]", n, EC_MAXN);
  float *lam, *G;
  const Tri T = lay_out(work, n, lam, G);
  float* za = static_cast<float*>(work2);
  float* zb = za + (size_t)n * n;
  tridiag(Load128{A, n}, n, T, s);
  k_tri_vectors<<<(n + TV_WARPS - 1) / TV_WARPS, 32 * TV_WARPS, 0, s>>>(T, n, lam, za);
  KS_CHECK_LAUNCH();
  k_tri_degenerate<<<1, 32 * DG_WARPS, 0, s>>>(T, n, lam, za);
  KS_CHECK_LAUNCH();
  const dim3 tiles((n + 31) / 32, (n + 31) / 32);
  for (int it = 0; it < NS_STEPS; ++it) {
    k_ns_gram<<<tiles, 256, 0, s>>>(za, n, G, T.nserr + it);
    KS_CHECK_LAUNCH();
    k_ns_update<<<tiles, 256, 0, s>>>(za, G, n, T.nserr + it, zb);
    KS_CHECK_LAUNCH();
    std::swap(za, zb);
  }
  k_back_transform<<<(n + BK_WARPS - 1) / BK_WARPS, 32 * BK_WARPS, 0, s>>>(T, n, za, V);
  KS_CHECK_LAUNCH();
}

void rr_step_mixed(const float2* Hraw, const float2* M, double alpha, int n, float2* Mcat, float2* Aout,
                   float2* Vout, int* perm, void* work, cudaStream_t s) {
  if (n > RR_MAXN || n < 1) fail(KS_ERR_ARG, "rr_step_mixed: n=%d not in [1, %d]", n, RR_MAXN);
  if (n <= SMALL_SUBSPACE) {
    rr_step_small(Hraw, M, alpha, n, Mcat, Aout, Vout, perm, s);
    return;
  }
  float *lam, *G;
  const Tri T = lay_out(work, n, lam, G);
  float* zt = reinterpret_cast<float*>(Mcat);                        // [n][n] floats, read before Mcat is written
  const dim3 tiles((n + 31) / 32, (n + 31) / 32);
  k_rr_product<0><<<tiles, 256, 0, s>>>(Hraw, M, n, MatOut{Vout, nullptr, nullptr, 0.f, nullptr});
  KS_CHECK_LAUNCH();
  k_rr_product<1><<<tiles, 256, 0, s>>>(M, Vout, n, MatOut{Aout, nullptr, nullptr, 0.f, nullptr});
  KS_CHECK_LAUNCH();
  tridiag(LoadPart{Aout, n}, n, T, s);
  k_tri_vectors<<<(n + TV_WARPS - 1) / TV_WARPS, 32 * TV_WARPS, 0, s>>>(T, n, lam, zt);
  KS_CHECK_LAUNCH();
  k_tri_degenerate<<<1, 32 * DG_WARPS, 0, s>>>(T, n, lam, zt);
  KS_CHECK_LAUNCH();
  k_back_transform<<<(n + BK_WARPS - 1) / BK_WARPS, 32 * BK_WARPS, 0, s>>>(T, n, zt, Vout);
  KS_CHECK_LAUNCH();
  k_rr_product<2><<<tiles, 256, 0, s>>>(Vout, M, n, MatOut{nullptr, Mcat, lam, (float)alpha, perm});
  KS_CHECK_LAUNCH();
}

void ritz_values(const float2* A, const float2* V, const int* perm, int n, double* eig, cudaStream_t s) {
  if (n > RR_MAXN || n < 1) fail(KS_ERR_ARG, "ritz_values: n=%d not in [1, %d]", n, RR_MAXN);
  k_ritz_values<<<n, 256, 0, s>>>(A, V, perm, n, eig);
  KS_CHECK_LAUNCH();
}

}  // namespace ks
