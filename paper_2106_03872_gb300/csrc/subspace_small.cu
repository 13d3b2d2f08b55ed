// Subspace kernels for blocks of at most 16 states on the mixed path: the eigensolver, the whole
// Rayleigh-Ritz step and the Cholesky factor, in one CTA each.  The chain of dependent steps bounds them; at
// these sizes the launches of the spread-out solver (eigh.cu) cost more than its parallelism saves: kernel time of
// a Rayleigh-Ritz step 19 us at 8 and 37 us at 16 states in one launch, where seven launches take 54 us at 17; of
// the eigensolver 20 and 36 us, where ten take 60 us.
//
// The eigensolver, FP32, matrix in shared memory, a warp per row:
//   1. Householder reduction to a real symmetric tridiagonal T, the update of step k-1 applied in the
//      same pass over the trailing block as the product A v_k of step k (one barrier a step; every warp
//      forms v_k itself from column k).
//   2. T is split where an off-diagonal element is negligible; eigenvalues by multisection on the Sturm
//      count (8 lanes per eigenvalue).
//   3. Vectors by twisted factorisation; inverse iteration with Gram-Schmidt inside numerically
//      degenerate clusters; Newton-Schulz steps (not in the Rayleigh-Ritz step).
//   4. Back-transformation, 8 threads per column.
// The Rayleigh-Ritz step adds H_sub = conj(M) H_raw M^T before and the step matrix after, as
// rr_step_mixed does (eigh.cu).
#include "kernels.h"

namespace ks {

namespace {

constexpr int EH_MAXN = SMALL_SUBSPACE;
constexpr int EH_THREADS = 512;                                      // a warp per row of the matrix
constexpr int EH_WARPS = EH_THREADS / 32;
static_assert(EH_MAXN <= EH_WARPS && EH_MAXN <= 32, "a warp per row, a lane per column");
constexpr unsigned FULL = 0xffffffffu;
// shared memory: the matrix [n][n + 1], then packed reflectors or three staged n x n operands
constexpr int EH_AREG = EH_MAXN * (EH_MAXN + 1);
constexpr int EH_RREG = 3 * EH_MAXN * EH_MAXN;
constexpr int SC_THREADS = 256;

__device__ __forceinline__ float2 cm(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 cmc(float2 a, float2 b) {   // conj(a) * b
  return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 cfma(float2 acc, float2 a, float2 b) {   // acc + a b
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(-a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(a.y, b.x, acc.y);
  return acc;
}
__device__ __forceinline__ float2 cfmac(float2 acc, float2 a, float2 b) {  // acc + conj(a) b
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(-a.y, b.x, acc.y);
  return acc;
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 warp_sum(float2 v) {
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(FULL, v.x, o);
    v.y += __shfl_xor_sync(FULL, v.y, o);
  }
  return v;
}

// Number of eigenvalues of T[b0..b1] below x (Sturm count of the LDL^T pivots).
__device__ __forceinline__ int sturm_count(const float* d, const float* e2, int b0, int b1, float x, float pivmin) {
  int c = 0;
  float q = d[b0] - x;
  if (fabsf(q) < pivmin) q = -pivmin;
  c += q < 0.f;
  for (int i = b0 + 1; i <= b1; ++i) {
    q = d[i] - x - __fdividef(e2[i - 1], q);
    if (fabsf(q) < pivmin) q = -pivmin;
    c += q < 0.f;
  }
  return c;
}

// A = conj(M) H_raw M^T (FP32), its Hermitian part, in the [n][n + 1] matrix region, and to Aout.  R stages
// H_raw, M (lower triangular, zeros stored) and H_raw M^T; each sum runs over k in ascending order.
__device__ __forceinline__ void subspace_matrix_small(const float2* __restrict__ Hraw, const float2* __restrict__ M, int n,
                                                float2* A, float2* R, float2* __restrict__ Aout) {
  const int ld = n + 1, t = threadIdx.x, i = t / n, j = t - i * n;
  const bool in = t < n * n;
  float2 *Hs = R, *Ms = Hs + EH_MAXN * EH_MAXN, *Ts = Ms + EH_MAXN * EH_MAXN;
  if (in) {
    Hs[t] = Hraw[t];
    Ms[t] = M[t];
  }
  __syncthreads();
  float2 acc = make_float2(0.f, 0.f);
  if (in) {
    for (int k = 0; k < n; ++k) acc = cfma(acc, Hs[i * n + k], Ms[j * n + k]);
    Ts[t] = acc;
  }
  __syncthreads();
  acc = make_float2(0.f, 0.f);
  if (in) {
    for (int k = 0; k < n; ++k) acc = cfmac(acc, Ms[i * n + k], Ts[k * n + j]);
    A[i * ld + j] = acc;
  }
  __syncthreads();
  float2 h = acc;
  if (in) {                                                          // Hermitian part, real diagonal
    const float2 b = A[j * ld + i];
    h = make_float2(0.5f * (acc.x + b.x), i == j ? 0.f : 0.5f * (acc.y - b.y));
  }
  __syncthreads();
  if (in) {
    A[i * ld + j] = h;
    Aout[t] = h;
  }
}

// With the vectors V in the matrix region (V_kr at k ld + r): C = Vt M (C_rj = sum_k V_kr M_kj, k ascending) and
// Mcat row rank(r) = [(1 + alpha lam_r) C_r | -alpha C_r].
__device__ __forceinline__ void step_matrix_small(const float2* Vs, const float2* __restrict__ M, int n, const float* lam,
                                            const int* rank, float alpha, float2* R, float2* __restrict__ Mcat) {
  const int ld = n + 1, t = threadIdx.x, r = t / n, j = t - r * n;
  if (t < n * n) R[t] = M[t];
  __syncthreads();
  if (t >= n * n) return;
  float2 c = make_float2(0.f, 0.f);
  for (int k = 0; k < n; ++k) c = cfma(c, Vs[k * ld + r], R[k * n + j]);
  const float f = 1.f + alpha * lam[r];
  float2* row = Mcat + (size_t)rank[r] * 2 * n;
  row[j] = make_float2(f * c.x, f * c.y);
  row[n + j] = make_float2(-alpha * c.x, -alpha * c.y);
}

// Inputs and outputs of the Rayleigh-Ritz variant (all device pointers, row-major, FP32).
struct RRStep {
  const float2* Hraw;   // [n][n] Psi^H (H Psi)
  const float2* M;      // [n][n] lower-triangular orthonormaliser
  float alpha;          // steepest-descent step
  float2* Mcat;         // [n][2n] step matrix
  float2* Aout;         // [n][n] Hermitian subspace matrix
  float2* Vout;         // [n][n] eigenvectors, column j for lam_j (unsorted)
  int* perm;            // [n] rank of lam_j
};

template <bool RR>
__global__ void __launch_bounds__(EH_THREADS, 1)
    k_eigh_small(const double2* __restrict__ H, int n, double2* __restrict__ Vout, RRStep rr) {
  __shared__ __align__(16) float2 A[EH_AREG];                        // [n][ld]
  __shared__ float2 R[EH_RREG];                                      // packed reflectors
  __shared__ float d[EH_MAXN], e[EH_MAXN], e2[EH_MAXN], lam[EH_MAXN];
  __shared__ float2 tau[EH_MAXN], wvp[2][EH_MAXN], red[2][32];
  __shared__ int blk_lo[EH_MAXN], blk_hi[EH_MAXN];
  __shared__ float s_err[EH_WARPS];
  const int ld = n + 1;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;

  if (t < 64) red[t >> 5][t & 31] = make_float2(0.f, 0.f);           // entries without a warp stay zero
  if constexpr (RR) {
    subspace_matrix_small(rr.Hraw, rr.M, n, A, R, rr.Aout);
  } else {
    for (int idx = t; idx < n * n; idx += EH_THREADS) {
      const int i = idx / n, j = idx - (idx / n) * n;
      const double2 h = H[idx];
      A[i * ld + j] = make_float2((float)h.x, i == j ? 0.f : (float)h.y);
    }
  }
  __syncthreads();

  // ---- 1. tridiagonalization ---------------------------------------------------------------
  // Entering step k, A[k:, k:] holds the updates of steps < k-1; the update of step k-1
  // (v_{k-1} at R + rprev, w_{k-1} = wvp[(k-1)&1] + ap v_{k-1}) is still to be applied.
  // A lane owns row / column j = k+1+lane, a warp row k+1+warp.
  int rprev = 0, roff = 0;
  for (int k = 0; k + 1 < n; ++k) {
    const int m = n - k - 1;
    const bool hp = k > 0;
    const int pb = (k + 1) & 1;                                     // buffer of step k-1
    const int j = k + 1 + lane, i = k + 1 + warp;
    const float2 zero = make_float2(0.f, 0.f);
    float2 ap = zero;
    if (hp) {
      const float2 s = warp_sum(red[pb][lane]);
      const float2 h = cm(tau[k - 1], s);
      ap = make_float2(-0.5f * h.x, -0.5f * h.y);
    }
    // pending-update vectors at the lane's index and at k
    float2 vp = zero, wp = zero;
    if (hp && j < n) {
      vp = R[rprev + j - k];
      wp = cadd(wvp[pb][j], cm(ap, vp));
    }
    const float2 wk = hp ? cadd(wvp[pb][k], ap) : zero;              // v_{k-1}[k] = 1
    // column k after the pending update: x_j = A_jk - (v_j conj(w_k) + w_j)
    float2 x = zero;
    float xn2 = 0.f;
    if (j < n) {
      const float2 u = cadd(make_float2(vp.x * wk.x + vp.y * wk.y, vp.y * wk.x - vp.x * wk.y), wp);
      x = csub(A[j * ld + k], u);
      if (lane > 0) xn2 = x.x * x.x + x.y * x.y;
    }
    for (int o = 16; o > 0; o >>= 1) xn2 += __shfl_xor_sync(FULL, xn2, o);
    const float2 al = make_float2(__shfl_sync(FULL, x.x, 0), __shfl_sync(FULL, x.y, 0));
    float2 tk, sc = zero;
    float ek;
    const float s2 = al.x * al.x + al.y * al.y + xn2;
    if (xn2 == 0.f && al.y == 0.f) {
      tk = zero;
      ek = al.x;
    } else if (s2 < 1e-30f) {
      // a column already reduced up to rounding noise (|x| < 1e-15): no reflection and a zero
      // off-diagonal element, which moves eigenvalues by < 1e-15; forming the reflector from
      // such a column would underflow its squares and divide by zero
      tk = zero;
      ek = 0.f;
    } else {
      const float beta = -copysignf(sqrtf(al.x * al.x + al.y * al.y + xn2), al.x);
      const float rb = __frcp_rn(beta);
      tk = make_float2((beta - al.x) * rb, -al.y * rb);
      const float2 dn = make_float2(al.x - beta, al.y);            // 1 / (alpha - beta)
      const float inv = __frcp_rn(dn.x * dn.x + dn.y * dn.y);
      sc = make_float2(dn.x * inv, -dn.y * inv);
      ek = beta;
    }
    const float2 vk = lane == 0 ? make_float2(1.f, 0.f) : (j < n ? cm(x, sc) : zero);
    if (warp == 0) {
      if (j < n) R[roff + lane] = vk;
      if (lane == 0) {
        tau[k] = tk;
        e[k] = ek;
        d[k] = A[k * ld + k].x - 2.f * wk.x;
      }
    }
    // trailing block: apply the update of step k-1 to row i, then w'_i = tau_k sum_j A_ij v_j
    float2 acc = zero;
    if (i < n) {                                                     // warp-uniform
      float2 vi = zero, wi = zero;
      if (hp) {
        vi = R[rprev + i - k];
        wi = cadd(wvp[pb][i], cm(ap, vi));
      }
      if (j < n) {
        float2 a = A[i * ld + j];
        if (hp) {
          // v_i conj(w_j) + w_i conj(v_j)
          a.x -= (vi.x * wp.x + vi.y * wp.y) + (wi.x * vp.x + wi.y * vp.y);
          a.y -= (vi.y * wp.x - vi.x * wp.y) + (wi.y * vp.x - wi.x * vp.y);
        }
        if (i == j) a.y = 0.f;
        A[i * ld + j] = a;
        acc = make_float2(a.x * vk.x - a.y * vk.y, a.x * vk.y + a.y * vk.x);
      }
    }
    acc = warp_sum(acc);
    // v_k at row i lives in lane i - k - 1 = warp
    const float2 vr = make_float2(__shfl_sync(FULL, vk.x, warp), __shfl_sync(FULL, vk.y, warp));
    float2 pw = zero;
    if (i < n) {
      const float2 w = cm(tk, acc);
      if (lane == 0) wvp[k & 1][i] = w;
      pw = cmc(w, vr);
    }
    if (lane == 0) red[k & 1][warp] = pw;
    rprev = roff;
    roff += m;
    __syncthreads();
  }
  if (t == 0) {
    if (n >= 2) {
      // last pending update (v_{n-2} = (1)), then d_{n-1}
      float2 s = make_float2(0.f, 0.f);
      for (int w = 0; w < EH_WARPS; ++w) s = cadd(s, red[n & 1][w]);
      const float2 h = cm(tau[n - 2], s);
      const float wl = wvp[n & 1][n - 1].x - 0.5f * h.x;
      d[n - 1] = A[(n - 1) * ld + (n - 1)].x - 2.f * wl;
    } else {
      d[0] = A[0].x;
    }
    e[n - 1] = 0.f;
  }
  __syncthreads();

  // ---- 2. split and eigenvalues ------------------------------------------------------------
  if (t == 0) {
    // blocks: e[i] negligible against its neighbours -> boundary after i
    int b0 = 0;
    for (int i = 0; i < n; ++i) {
      const bool cut = (i == n - 1) || fabsf(e[i]) <= 1e-7f * (fabsf(d[i]) + fabsf(d[i + 1]) + 1e-30f);
      if (cut) {
        for (int j = b0; j <= i; ++j) {
          blk_lo[j] = b0;
          blk_hi[j] = i;
        }
        if (i < n - 1) e[i] = 0.f;
        b0 = i + 1;
      }
    }
    for (int i = 0; i < n; ++i) e2[i] = e[i] * e[i];
  }
  __syncthreads();
  float tnorm = 0.f;
  for (int i = 0; i < n; ++i) tnorm = fmaxf(tnorm, fabsf(d[i]) + fabsf(e[i]) + (i > 0 ? fabsf(e[i - 1]) : 0.f));
  {
    // slot = t / 8 (one eigenvalue), 8 lanes evaluate 8 interior points of the interval
    const int slot = t >> 3, sub = t & 7;
    const bool active = slot < n;
    int b0 = 0, b1 = 0, kth = 0;
    float lo = 0.f, hi = 0.f;
    if (active) {
      b0 = blk_lo[slot];
      b1 = blk_hi[slot];
      kth = slot - b0;
      lo = 1e30f;
      hi = -1e30f;
      for (int i = b0; i <= b1; ++i) {
        const float r = (i > b0 ? fabsf(e[i - 1]) : 0.f) + (i < b1 ? fabsf(e[i]) : 0.f);
        lo = fminf(lo, d[i] - r);
        hi = fmaxf(hi, d[i] + r);
      }
      const float pad = 1e-6f * fmaxf(fabsf(lo), fabsf(hi)) + 1e-20f;
      lo -= pad;
      hi += pad;
    }
    const float width = 4.8e-7f * tnorm + 1e-30f;                    // ~4 ulps of |T|
    for (int iter = 0; iter < 24; ++iter) {
      const bool need = active && (hi - lo > width);
      if (!__any_sync(FULL, need)) break;
      const float x = lo + (hi - lo) * (float)(sub + 1) * (1.f / 9.f);
      const int c = need ? sturm_count(d, e2, b0, b1, x, 1e-30f) : 0;
      // new lo: largest x with count <= kth; new hi: smallest x with count >= kth + 1
      float nlo = (need && c <= kth) ? x : -1e30f;
      float nhi = (need && c >= kth + 1) ? x : 1e30f;
      for (int o = 4; o > 0; o >>= 1) {
        nlo = fmaxf(nlo, __shfl_xor_sync(FULL, nlo, o));
        nhi = fminf(nhi, __shfl_xor_sync(FULL, nhi, o));
      }
      if (nlo > lo) lo = nlo;
      if (nhi < hi) hi = nhi;
    }
    if (active && sub == 0) lam[slot] = 0.5f * (lo + hi);
  }
  __syncthreads();

  // ---- 3. eigenvectors of T ----------------------------------------------------------------
  // Z (real, [n][zld]) in the second half of the A region; D- pivots [n][n] and later
  // Z^T Z in the first.
  const int zld = n + 1;
  const float tiny = 1e-30f + 1e-13f * tnorm;                        // pivot floor
  float* low = reinterpret_cast<float*>(A);
  float* Zr = low + EH_MAXN * EH_MAXN;
  static_assert(EH_MAXN * EH_MAXN + EH_AREG <= 2 * EH_AREG, "both fit");
  for (int idx = t; idx < n * zld; idx += EH_THREADS) Zr[idx] = 0.f;
  __syncthreads();
  if (t < n) {
    const int slot = t;
    const int b0 = blk_lo[slot], b1 = blk_hi[slot];
    const float x = lam[slot];
    if (b0 == b1) {
      Zr[b0 * zld + slot] = 1.f;
    } else {
      // backward pivots D-: dm_i = d_i - x - e_i^2 / dm_{i+1}, kept in low[i][slot]
      float q = d[b1] - x;
      if (fabsf(q) < tiny) q = tiny;
      low[b1 * n + slot] = q;
      for (int i = b1 - 1; i >= b0; --i) {
        q = d[i] - x - __fdividef(e2[i], q);
        if (fabsf(q) < tiny) q = tiny;
        low[i * n + slot] = q;
      }
      // forward pivots D+ with gamma_i = dp_i + dm_i - (d_i - x); the ratios -e_i / dp_i
      // go to Z's column until the twist index r (argmin |gamma|) is known
      int r = b0;
      float best = 3.4e38f;
      q = d[b0] - x;
      if (fabsf(q) < tiny) q = tiny;
      for (int i = b0; i <= b1; ++i) {
        if (i > b0) {
          q = d[i] - x - __fdividef(e2[i - 1], q);
          if (fabsf(q) < tiny) q = tiny;
        }
        const float g = fabsf(q + low[i * n + slot] - (d[i] - x));
        if (g < best) {
          best = g;
          r = i;
        }
        if (i < b1) Zr[i * zld + slot] = -__fdividef(e[i], q);
      }
      float nrm = 1.f, z = 1.f;
      for (int i = r - 1; i >= b0; --i) {
        z *= Zr[i * zld + slot];
        Zr[i * zld + slot] = z;
        nrm += z * z;
      }
      Zr[r * zld + slot] = 1.f;
      z = 1.f;
      for (int i = r + 1; i <= b1; ++i) {
        z *= -__fdividef(e[i - 1], low[i * n + slot]);
        Zr[i * zld + slot] = z;
        nrm += z * z;
      }
      const float inv = rsqrtf(nrm);
      for (int i = b0; i <= b1; ++i) Zr[i * zld + slot] *= inv;
    }
  }
  __syncthreads();
  // Degenerate clusters of a block (lam gaps <= 1e-5 |T|): twisted factorization returns
  // (nearly) the same vector for every member, so each member after the first is recomputed
  // by inverse iteration -- two LDL^T solves of (T - lam_j) y = x from a pseudo-random start,
  // each followed by Gram-Schmidt against the earlier members of the cluster (the scheme of
  // LAPACK's stein).  One warp per block; lane 0 runs the serial solves.
  for (int b = warp; b < n; b += EH_WARPS) {
    if (blk_lo[b] != b) continue;
    const int b1 = blk_hi[b];
    float* Lc = low + warp * EH_MAXN;                                // L's subdiagonal
    for (int j = b + 1; j <= b1; ++j) {
      int c0 = j;
      while (c0 > b && lam[c0] - lam[c0 - 1] <= 1e-5f * tnorm) --c0;
      if (c0 == j) continue;
      for (int i = b + lane; i <= b1; i += 32) {
        const unsigned hsh = (unsigned)(i * 131 + j * 7919) * 2654435761u;
        Zr[i * zld + j] = (float)(hsh >> 16) * (1.f / 32768.f) - 1.f;
      }
      __syncwarp();
      const float lj = lam[j];
      for (int it = 0; it < 2; ++it) {
        if (lane == 0) {
          float piv = d[b] - lj;
          if (fabsf(piv) < tiny) piv = tiny;
          float u = Zr[b * zld + j];
          Zr[b * zld + j] = __fdividef(u, piv);
          for (int i = b + 1; i <= b1; ++i) {
            const float l = __fdividef(e[i - 1], piv);
            Lc[i - 1] = l;
            piv = d[i] - lj - l * e[i - 1];
            if (fabsf(piv) < tiny) piv = tiny;
            u = Zr[i * zld + j] - l * u;
            Zr[i * zld + j] = __fdividef(u, piv);
          }
          for (int i = b1 - 1; i >= b; --i) Zr[i * zld + j] -= Lc[i] * Zr[(i + 1) * zld + j];
        }
        __syncwarp();
        for (int p = c0; p < j; ++p) {
          float sd = 0.f;
          for (int i = b + lane; i <= b1; i += 32) sd += Zr[i * zld + p] * Zr[i * zld + j];
          for (int o = 16; o > 0; o >>= 1) sd += __shfl_xor_sync(FULL, sd, o);
          for (int i = b + lane; i <= b1; i += 32) Zr[i * zld + j] -= sd * Zr[i * zld + p];
          __syncwarp();
        }
        float sn = 0.f;
        for (int i = b + lane; i <= b1; i += 32) sn += Zr[i * zld + j] * Zr[i * zld + j];
        for (int o = 16; o > 0; o >>= 1) sn += __shfl_xor_sync(FULL, sn, o);
        const float inv = rsqrtf(fmaxf(sn, 1e-30f));
        for (int i = b + lane; i <= b1; i += 32) Zr[i * zld + j] *= inv;
        __syncwarp();
      }
    }
  }
  __syncthreads();
  // Newton-Schulz: G = Z^T Z; while max |G - I| > 2e-6: Z <- 1.5 Z - 0.5 Z G.
  // Thread: row warp, column lane.  The Rayleigh-Ritz variant skips it: its vectors only span the next
  // iterate, whose CholQR orthonormalises the block, and outside degenerate clusters (handled above) they
  // are orthogonal to eps |T| / gap <= 6e-3, a condition number of the step matrix within 1.01.
  if constexpr (!RR) {
    float* G = low;                                                  // [n][n]
    const bool in = warp < n && lane < n;
    for (int it = 0; it < 4; ++it) {
      float g = 0.f, err = 0.f;
      if (in) {
        for (int i = 0; i < n; ++i) g += Zr[i * zld + warp] * Zr[i * zld + lane];
        G[warp * n + lane] = g;
        err = fabsf(g - (warp == lane ? 1.f : 0.f));
      }
      for (int o = 16; o > 0; o >>= 1) err = fmaxf(err, __shfl_xor_sync(FULL, err, o));
      if (lane == 0) s_err[warp] = err;
      __syncthreads();
      float emax = 0.f;
      for (int w = 0; w < EH_WARPS; ++w) emax = fmaxf(emax, s_err[w]);
      if (!(emax > 2e-6f)) break;                                    // uniform
      float z = 0.f;
      if (in)
        for (int b = 0; b < n; ++b) z += Zr[warp * zld + b] * G[b * n + lane];
      __syncthreads();
      if (in) Zr[warp * zld + lane] = 1.5f * Zr[warp * zld + lane] - 0.5f * z;
      __syncthreads();
    }
  }

  // ---- 4. V = H_0 ... H_{n-2} Z ------------------------------------------------------------
  // thread (column j = t / 8, s = t % 8) holds rows s + 8p, p < 2.  The reflectors are
  // expanded into a zero-padded [n-1][EH_MAXN] layout in the A region (v_k[i] = 0 for i <= k
  // and i >= n), so no row needs a bounds test.
  {
    const int j = t >> 3, s = t & 7;
    float2 V[EH_MAXN / 8];
#pragma unroll
    for (int p = 0; p < EH_MAXN / 8; ++p) {
      const int i = s + 8 * p;
      V[p] = make_float2((i < n && j < n) ? Zr[i * zld + j] : 0.f, 0.f);
    }
    __syncthreads();
    float2* Rf = A;
    for (int idx = t; idx < (n - 1) * EH_MAXN; idx += EH_THREADS) {
      const int k = idx / EH_MAXN, i = idx - k * EH_MAXN;
      const int ro = k * (n - 1) - (k * (k - 1)) / 2;
      Rf[idx] = (i > k && i < n) ? R[ro + i - k - 1] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int k = n - 2; k >= 0; --k) {
      const float2 tk = tau[k];
      if (tk.x == 0.f && tk.y == 0.f) continue;                      // uniform
      const float2* v = Rf + k * EH_MAXN + s;                        // v[8p] = v_k at row s + 8p
      const int pskip = (k + 1) >> 3;                                // rows s + 8p < k+1 below
      float2 dot = make_float2(0.f, 0.f);
#pragma unroll
      for (int p = 0; p < EH_MAXN / 8; ++p) {
        if (p >= pskip) {
          const float2 c = cmc(v[8 * p], V[p]);
          dot.x += c.x;
          dot.y += c.y;
        }
      }
      for (int o = 4; o > 0; o >>= 1) {
        dot.x += __shfl_xor_sync(FULL, dot.x, o);
        dot.y += __shfl_xor_sync(FULL, dot.y, o);
      }
      const float2 c = cm(tk, dot);
#pragma unroll
      for (int p = 0; p < EH_MAXN / 8; ++p)
        if (p >= pskip) V[p] = csub(V[p], cm(v[8 * p], c));
    }
    // stage through shared memory (the A region) for coalesced complex128 stores
    __syncthreads();
    float2* Vs = A;                                                  // [n][ld]
    if (j < n) {
#pragma unroll
      for (int p = 0; p < EH_MAXN / 8; ++p) {
        const int i = s + 8 * p;
        if (i < n) Vs[i * ld + j] = V[p];
      }
    }
  }
  __syncthreads();
  if constexpr (RR) {
    // ranks of the eigenvalues (ties by index) and the exported vectors
    int* rank = blk_lo;
    if (t < n) {
      const float li = lam[t];
      int r = 0;
      for (int j = 0; j < n; ++j) r += (lam[j] < li) || (lam[j] == li && j < t);
      rank[t] = r;
      rr.perm[t] = r;
    }
    for (int i = warp; i < n; i += EH_WARPS)
      for (int j = lane; j < n; j += 32) rr.Vout[i * n + j] = A[i * ld + j];
    __syncthreads();
    step_matrix_small(A, rr.M, n, lam, rank, rr.alpha, R, rr.Mcat);
  } else {
    for (int idx = t; idx < n * n; idx += EH_THREADS) {
      const int i = idx / n, j = idx - (idx / n) * n;
      const float2 v = A[i * ld + j];
      Vout[idx] = make_double2((double)v.x, (double)v.y);
    }
  }
}

// One CTA.  Reads the lower triangle of S (n x n, row-major), writes X = L^{-1} (lower,
// zeros above; conj(X) when conj_out) to Out, and an FP32 copy to Out32 when it is given.
//
// Shared memory holds one square [n][ld] array: L_rc (r >= c) at [c][r] (column-major, so
// lanes running along a column touch consecutive words) and X_rc (r > c) at [r][c], i.e. in
// the unused upper triangle; X's diagonal is a separate vector.  Blocked by CB columns, each
// block step three barriers:
//   (a) warp 0 factors the diagonal block in registers (lane = row, the pivot column is
//       broadcast by shuffles) and inverts it in registers;
//   (b) panel L_iJ = A_iJ W_J^H for the rows below (all threads);
//   (c) trailing update A_ik -= sum_{c in J} L_ic conj(L_kc) (warps over columns k, lanes
//       over rows i; conj(L_kJ) held in registers).
// Then the off-diagonal blocks of X by block rows I: T_IJ = sum_{K=J}^{I-1} L_IK X_KJ,
// X_IJ = -W_I T_IJ for all J < I at once.
constexpr int CB = 8;

__device__ __forceinline__ float2 c_mul(float2 a, float2 b) { return cm(a, b); }
__device__ __forceinline__ float2 c_mulc(float2 a, float2 b) {   // a * conj(b)
  return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
__device__ __forceinline__ float2 shfl2(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

__global__ void __launch_bounds__(SC_THREADS, 1)
    k_chol_small(const double2* __restrict__ S, int n, double tol, int conj_out, int* __restrict__ status,
                 double2* __restrict__ Out, float2* __restrict__ Out32) {
  constexpr int MAXN = SMALL_SUBSPACE;
  __shared__ float2 U[MAXN * (MAXN + 1)];
  const int ld = n + 1;
  __shared__ float sjj[MAXN];
  __shared__ float2 xd[MAXN];                                        // diagonal of X
  __shared__ int s_bad;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  constexpr int NW = SC_THREADS / 32;
#define UL(r, c) U[(c) * ld + (r)]
#define XU(r, c) U[(r) * ld + (c)]
#define XL(r, c) ((r) == (c) ? xd[r] : XU(r, c))

  for (int e = t; e < n * n; e += SC_THREADS) {
    const int r = e / n, c = e - (e / n) * n;
    if (c <= r) {
      const double2 v = S[e];
      UL(r, c) = make_float2((float)v.x, r == c ? 0.f : (float)v.y);
    }
  }
  for (int j = t; j < n; j += SC_THREADS) sjj[j] = (float)S[(size_t)j * n + j].x;
  if (t == 0) s_bad = 0;
  __syncthreads();

  for (int J = 0; J < n; J += CB) {
    const int jb = min(CB, n - J), J1 = J + jb;
    // (a) diagonal block in warp 0's registers: lane r holds row J + r
    if (warp == 0) {
      float2 a[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) a[c] = (c <= lane && lane < jb) ? UL(J + lane, J + c) : make_float2(0.f, 0.f);
      int bad = 0;
#pragma unroll
      for (int j = 0; j < CB; ++j) {
        if (j < jb && !bad) {
          const float d = __shfl_sync(0xffffffffu, a[j].x, j);
          if (!(d > (float)tol * sjj[J + j]) || !isfinite(d)) {
            bad = J + j + 1;
          } else {
            const float ljj = sqrtf(d), inv = 1.f / ljj;
            if (lane == j) a[j] = make_float2(ljj, 0.f);
            else if (lane > j) a[j] = make_float2(a[j].x * inv, a[j].y * inv);
#pragma unroll
            for (int k = j + 1; k < CB; ++k) {
              const float2 lkj = shfl2(a[j], k);
              if (k <= lane) {
                const float2 p = c_mulc(a[j], lkj);
                a[k].x -= p.x;
                a[k].y -= p.y;
              }
            }
          }
        }
      }
      if (bad) {
        if (lane == 0) s_bad = bad;
      } else {
#pragma unroll
        for (int c = 0; c < CB; ++c)
          if (c <= lane && lane < jb) UL(J + lane, J + c) = a[c];
        // W = L_JJ^{-1} by rows: row j final after division by L_jj, rows r > j lose L_rj W_j
        float2 w[CB];
#pragma unroll
        for (int c = 0; c < CB; ++c) w[c] = make_float2(c == lane ? 1.f : 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < CB; ++j) {
          if (j < jb) {
            const float ij = 1.f / __shfl_sync(0xffffffffu, a[j].x, j);
            if (lane == j) {
#pragma unroll
              for (int c = 0; c <= j; ++c) w[c] = make_float2(w[c].x * ij, w[c].y * ij);
            }
#pragma unroll
            for (int c = 0; c <= j; ++c) {
              const float2 wj = shfl2(w[c], j);
              if (lane > j) {
                const float2 p = c_mul(a[j], wj);
                w[c].x -= p.x;
                w[c].y -= p.y;
              }
            }
          }
        }
        if (lane < jb) {
#pragma unroll
          for (int c = 0; c < CB; ++c) {
            if (c < lane) XU(J + lane, J + c) = w[c];
            else if (c == lane) xd[J + lane] = w[c];
          }
        }
      }
    }
    __syncthreads();
    if (s_bad) break;                                                // uniform
    const int rows = n - J1;
    if (rows == 0) break;
    // (b) panel: L_ic = sum_{k=J}^{c} A_ik conj(W_ck); lanes run along i
    float2 pv[(MAXN * CB + SC_THREADS - 1) / SC_THREADS];
#pragma unroll
    for (int q = 0; q < (MAXN * CB + SC_THREADS - 1) / SC_THREADS; ++q) {
      const int idx = t + q * SC_THREADS;
      pv[q] = make_float2(0.f, 0.f);
      if (idx < rows * jb) {
        const int i = J1 + idx % rows, c = J + idx / rows;
        for (int k = J; k <= c; ++k) {
          const float2 p = c_mulc(UL(i, k), XL(c, k));
          pv[q].x += p.x;
          pv[q].y += p.y;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < (MAXN * CB + SC_THREADS - 1) / SC_THREADS; ++q) {
      const int idx = t + q * SC_THREADS;
      if (idx < rows * jb) UL(J1 + idx % rows, J + idx / rows) = pv[q];
    }
    __syncthreads();
    // (c) trailing update, columns k >= J1
    for (int k = J1 + warp; k < n; k += NW) {
      float2 lk[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const float2 v = c < jb ? UL(k, J + c) : make_float2(0.f, 0.f);
        lk[c] = make_float2(v.x, -v.y);
      }
      for (int i = k + lane; i < n; i += 32) {
        float2 acc = make_float2(0.f, 0.f);
        const float2* col = U + J * ld + i;                          // col[c * ld] = L_{i, J+c}
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          if (c < jb) {
            const float2 p = c_mul(col[c * ld], lk[c]);
            acc.x += p.x;
            acc.y += p.y;
          }
        }
        const float2 v = UL(i, k);
        UL(i, k) = make_float2(v.x - acc.x, v.y - acc.y);
      }
    }
    __syncthreads();
  }
  if (s_bad) {
    for (int e = t; e < n * n; e += SC_THREADS) {
      const bool diag = e / n == e % n;
      Out[e] = make_double2(diag ? 1.0 : 0.0, 0.0);
      if (Out32) Out32[e] = make_float2(diag ? 1.f : 0.f, 0.f);
    }
    if (t == 0) atomicCAS(status, 0, s_bad);
    return;
  }
  // off-diagonal blocks of X, block row by block row
  for (int I0 = CB; I0 < n; I0 += CB) {
    const int ib = min(CB, n - I0);
    // T_rc = sum_{k=c}^{I0-1} L_rk X_kc into X(r, c), r in block row I, c < I0 (lanes along r)
    for (int idx = t; idx < ib * I0; idx += SC_THREADS) {
      const int r = I0 + idx % ib, c = idx / ib;
      float2 acc = c_mul(UL(r, c), xd[c]);
      for (int k = c + 1; k < I0; ++k) {
        const float2 p = c_mul(UL(r, k), XU(k, c));
        acc.x += p.x;
        acc.y += p.y;
      }
      XU(r, c) = acc;
    }
    __syncthreads();
    // X_rc = -sum_{r'=I0}^{r} W_I[r][r'] T_r'c
    float2 xv[(CB * MAXN + SC_THREADS - 1) / SC_THREADS];
#pragma unroll
    for (int q = 0; q < (CB * MAXN + SC_THREADS - 1) / SC_THREADS; ++q) {
      const int idx = t + q * SC_THREADS;
      xv[q] = make_float2(0.f, 0.f);
      if (idx < ib * I0) {
        const int r = I0 + idx % ib, c = idx / ib;
        for (int rp = I0; rp <= r; ++rp) {
          const float2 p = c_mul(XL(r, rp), XU(rp, c));
          xv[q].x -= p.x;
          xv[q].y -= p.y;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < (CB * MAXN + SC_THREADS - 1) / SC_THREADS; ++q) {
      const int idx = t + q * SC_THREADS;
      if (idx < ib * I0) XU(I0 + idx % ib, idx / ib) = xv[q];
    }
    __syncthreads();
  }
  const float sgn = conj_out ? -1.f : 1.f;
  for (int e = t; e < n * n; e += SC_THREADS) {
    const int r = e / n, c = e - (e / n) * n;
    const float2 x = c <= r ? XL(r, c) : make_float2(0.f, 0.f);
    Out[e] = make_double2((double)x.x, (double)(sgn * x.y));
    if (Out32) Out32[e] = make_float2(x.x, sgn * x.y);
  }
#undef UL
#undef XU
#undef XL
}

}  // namespace

void eigh_small(const double2* A, double2* V, int n, cudaStream_t s) {
  if (n > SMALL_SUBSPACE || n < 1) fail(KS_ERR_ARG, "eigh_small: n=%d not in [1, %d]", n, SMALL_SUBSPACE);
  k_eigh_small<false><<<1, EH_THREADS, 0, s>>>(A, n, V, RRStep{});
  KS_CHECK_LAUNCH();
}

void rr_step_small(const float2* Hraw, const float2* M, double alpha, int n, float2* Mcat, float2* Aout,
                   float2* Vout, int* perm, cudaStream_t s) {
  if (n > SMALL_SUBSPACE || n < 1) fail(KS_ERR_ARG, "rr_step_small: n=%d not in [1, %d]", n, SMALL_SUBSPACE);
  const RRStep rr{Hraw, M, (float)alpha, Mcat, Aout, Vout, perm};
  k_eigh_small<true><<<1, EH_THREADS, 0, s>>>(nullptr, n, nullptr, rr);
  KS_CHECK_LAUNCH();
}

void chol32_small(const double2* S, int n, double tol, int conj_out, int* status, double2* Out, float2* Out32,
                  cudaStream_t s) {
  if (n > SMALL_SUBSPACE || n < 1) fail(KS_ERR_ARG, "chol32_small: n=%d not in [1, %d]", n, SMALL_SUBSPACE);
  k_chol_small<<<1, SC_THREADS, 0, s>>>(S, n, tol, conj_out, status, Out, Out32);
  KS_CHECK_LAUNCH();
}

}  // namespace ks
