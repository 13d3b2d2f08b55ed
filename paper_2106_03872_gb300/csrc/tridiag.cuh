// Householder reduction of a Hermitian FP32 matrix to real symmetric tridiagonal form by a cluster of
// CTAs (eigh.cu).
//
// The reflector H_k = I - tau_k v_k v_k^H (v_k[k+1] = 1) maps A[k+1:, k] to (beta_k, 0, ...) with real
// beta_k; the trailing block takes A -= v w^H + w v^H, w = w' - (tau/2)(w'^H v) v, w' = tau A v.  The
// update of step k-1 is applied in the same pass over the rows as the product A v_k of step k.
//
// What bounds it is the chain of n - 1 dependent steps, so a step holds as little as possible:
//   - the matrix lives in registers (row i in CTA i mod CL, a warp's NR rows, a lane's columns
//     lane + 32 q); out of shared memory its loads and stores alone took over 1000 cycles a step at
//     n = 128;
//   - one warp of each CTA forms the reflector (its part of the previous one stays in its registers);
//   - a warp's rows sum their products together (9 shuffles for four rows' complex sums, not 40);
//   - the rows' results are read from their owners' shared memory, one remote load per slot (written
//     to every CTA instead, the barrier waited for the stores: 630 to 1370 cycles a step);
//   - the steps are compiled once per 32-column slot of k, so that the slots and rows already reduced
//     drop out without branches (a warp-uniform branch around every slot cost more than it saved).
#pragma once

#include <cooperative_groups.h>

#include "common.h"

namespace ks {

template <int CL, int MAXN> struct TriShared {
  // g[k & 1][li] = (w'_i of step k-1, A_ik without that update) of this CTA's row i >= k at step k
  float4 g[2][MAXN / CL];
  float2 v[2][MAXN];     // v_k at [k & 1]
  float2 w[MAXN];        // w of step k-1
  float2 tau[MAXN];
  float d[MAXN], e[MAXN];
};

__device__ __forceinline__ float2 tri_mul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float tri_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// 1 / x and 1 / sqrt(x) for x in the normal range: the hardware approximation and one Newton step
__device__ __forceinline__ float tri_rcp(float x) {
  const float r = __fdividef(1.f, x);
  return fmaf(r, fmaf(-x, r, 1.f), r);
}
__device__ __forceinline__ float tri_rsqrt(float x) {
  const float r = rsqrtf(x);
  return fmaf(0.5f * r, fmaf(-x * r, r, 1.f), r);
}

// The sums over the warp of NV = 2, 4 or 8 values per lane: value q ends up in the lanes whose upper
// log2(NV) bits are q.
template <int NV> __device__ __forceinline__ float tri_sum_many(float (&v)[NV], int lane) {
  int o = 16;
#pragma unroll
  for (int h = NV / 2; h > 0; h /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int q = 0; q < h; ++q) {
      const float keep = up ? v[q + h] : v[q], give = up ? v[q] : v[q + h];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  float s = v[0];
#pragma unroll
  for (; o > 0; o /= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Where T, the reflectors and the flags of one decomposition live (global memory).
struct Tri {
  float* d;        // [n] diagonal
  float* e;        // [n] off-diagonal (e[n-1] = 0)
  float2* tau;     // [n]
  int* nserr;      // flags of the Newton-Schulz steps
  float2* R;       // [n-1][ldr] reflector k, zero up to column k (from the slot of k + 1 on) and from n on
  int ldr;         // n rounded up to a slot of 32
};

template <int CL, int THREADS, int MAXN> struct Tridiag {
  static constexpr int Q = MAXN / 32, NWARP = THREADS / 32, ML = MAXN / CL, NR = ML / NWARP;
  static constexpr int GL = 32 / NR;                                 // lanes of a row's group
  using Shared = TriShared<CL, MAXN>;
  static_assert(NR == 2 || NR == 4, "rows of a warp");
  static_assert(32 % CL == 0, "a lane's columns belong to one CTA");

  Shared& sh;
  const Tri& T;
  const float4* gsrc;    // where row j = lane + 32 q is published
  int n, rank, lane, warp;
  float2 A[NR][Q];
  float2 vp0[Q];         // warp 0: the previous reflector
  float2 tk;             // warp 0: its tau

  __device__ __forceinline__ static void barrier() {
    if constexpr (CL > 1)
      cooperative_groups::this_cluster().sync();
    else
      __syncthreads();
  }
  __device__ __forceinline__ int row(int r) const { return (warp + r * NWARP) * CL + rank; }

  __device__ __forceinline__ Tridiag(Shared& s, const Tri& t, int n_) : sh(s), T(t), n(n_) {
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    rank = 0;
    gsrc = &sh.g[0][0];
    if constexpr (CL > 1) {
      rank = (int)cooperative_groups::this_cluster().block_rank();
      gsrc = cooperative_groups::this_cluster().map_shared_rank(&sh.g[0][0], lane % CL);
    }
  }

  // Reflector k: zeros up to column k from the slot of k + 1 on, and from n on.
  __device__ __forceinline__ void store_reflector(int k, const float2* v) {
    for (int j = ((k + 1) & ~31) + lane; j < T.ldr; j += 32) T.R[(size_t)k * T.ldr + j] = v[j];
  }

  // Steps k with (k + 1) / 32 = Q1: slots below Q1 hold reduced columns, row groups below R1 reduced rows.
  template <int Q1> __device__ __forceinline__ void slot_steps() {
    constexpr int Q0 = Q1 > 0 ? Q1 - 1 : 0;                          // slot of column k at the first of them
    constexpr int R1 = Q1 * 32 / (NWARP * CL);
    const int k1 = min(32 * Q1 + 31, n - 1);
    for (int k = max(32 * Q1 - 1, 0); k < k1; ++k) {
      const int b = k & 1;
      if (warp == 0) {
        float2 wq[Q], a[Q];
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = Q0; q < Q; ++q) {
          const int j = lane + 32 * q;
          const float4 f = gsrc[b * ML + j / CL];
          const bool in = j >= k && j < n;                           // else not published at this step
          wq[q] = in ? make_float2(f.x, f.y) : make_float2(0.f, 0.f);
          a[q] = in ? make_float2(f.z, f.w) : make_float2(0.f, 0.f);
          s.x += wq[q].x * vp0[q].x + wq[q].y * vp0[q].y;            // conj(w') v
          s.y += wq[q].x * vp0[q].y - wq[q].y * vp0[q].x;
        }
        s.x = tri_sum(s.x);
        s.y = tri_sum(s.y);
        const float2 h = tri_mul(tk, s);
        const float2 ap = make_float2(-0.5f * h.x, -0.5f * h.y);
#pragma unroll
        for (int q = Q0; q < Q; ++q) {
          const float2 c = tri_mul(ap, vp0[q]);
          wq[q] = make_float2(wq[q].x + c.x, wq[q].y + c.y);
        }
        // w_k and A_kk: in slot Q1, or Q1 - 1 at the slot's first step
        const bool lower = Q1 > 0 && k < 32 * Q1;
        const float2 mk = lower ? wq[Q0] : wq[Q1];
        const float dk = (lower ? a[Q0].x : a[Q1].x) - 2.f * mk.x;   // lane of j = k: v_{k-1}[k] = 1
        const float2 wk = make_float2(__shfl_sync(0xffffffffu, mk.x, k & 31), __shfl_sync(0xffffffffu, mk.y, k & 31));
        // x_j = A_jk - (v_j conj(w_k) + w_j), j > k
        float xn2 = 0.f;
#pragma unroll
        for (int q = Q0; q < Q; ++q) {
          a[q].x -= vp0[q].x * wk.x + vp0[q].y * wk.y + wq[q].x;
          a[q].y -= vp0[q].y * wk.x - vp0[q].x * wk.y + wq[q].y;
          const float m = a[q].x * a[q].x + a[q].y * a[q].y;         // zero from n on
          xn2 += lane + 32 * q > k + 1 ? m : 0.f;
        }
        xn2 = tri_sum(xn2);
        const int la = (k + 1) & 31;
        const float2 al = make_float2(__shfl_sync(0xffffffffu, a[Q1].x, la), __shfl_sync(0xffffffffu, a[Q1].y, la));
        const float s2 = al.x * al.x + al.y * al.y + xn2;
        float2 sc = make_float2(0.f, 0.f);
        float ek = 0.f;
        tk = make_float2(0.f, 0.f);
        if (xn2 == 0.f && al.y == 0.f) {
          ek = al.x;
        } else if (!(s2 < 1e-30f)) {
          // (a column reduced to rounding noise, |x| < 1e-15, takes no reflection and a zero
          // off-diagonal element, which moves eigenvalues by < 1e-15: its squares would underflow)
          const float rs = tri_rsqrt(s2);
          const float beta = -copysignf(s2 * rs, al.x), rb = -copysignf(rs, al.x);
          tk = make_float2((beta - al.x) * rb, -al.y * rb);
          const float2 dn = make_float2(al.x - beta, al.y);
          const float inv = tri_rcp(dn.x * dn.x + dn.y * dn.y);
          sc = make_float2(dn.x * inv, -dn.y * inv);
          ek = beta;
        }
#pragma unroll
        for (int q = Q0; q < Q; ++q) {
          const int j = lane + 32 * q;
          float2 v = tri_mul(a[q], sc);
          v.x = j == k + 1 ? 1.f : (j <= k ? 0.f : v.x);
          v.y = j <= k + 1 ? 0.f : v.y;
          vp0[q] = v;
          sh.v[b][j] = v;
          sh.w[j] = wq[q];
        }
        if (lane == (k & 31)) {
          sh.tau[k] = tk;
          sh.e[k] = ek;
          sh.d[k] = dk;
        }
      } else if (warp == 1 && rank == 0 && k > 0) {
        // the previous reflector to global memory, early in the step: the cluster barrier at the
        // step's end waits for the stores in flight (950 cycles when they were issued late)
        store_reflector(k - 1, sh.v[b ^ 1]);
      }
      __syncthreads();
      // rows i > k: the pending update and the product with v_k.  Columns and rows <= k of the first
      // slots take values nothing reads again; v_k is zero there.
      float acc[2 * NR];
      float2 vi[NR], wi[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        acc[2 * r] = acc[2 * r + 1] = 0.f;
        if (r >= R1) {
          vi[r] = sh.v[b ^ 1][row(r)];
          wi[r] = sh.w[row(r)];
        }
      }
      float2 first[NR];                                              // A_{i,k+1} in its lane
#pragma unroll
      for (int q = Q1; q < Q; ++q) {
        const float2 v = sh.v[b][lane + 32 * q], vp = sh.v[b ^ 1][lane + 32 * q], wp = sh.w[lane + 32 * q];
#pragma unroll
        for (int r = R1; r < NR; ++r) {
          // v_i conj(w_c) + w_i conj(v_c)
          float2 m = A[r][q];
          m.x = fmaf(-vi[r].x, wp.x, fmaf(-vi[r].y, wp.y, fmaf(-wi[r].x, vp.x, fmaf(-wi[r].y, vp.y, m.x))));
          m.y = fmaf(-vi[r].y, wp.x, fmaf(vi[r].x, wp.y, fmaf(-wi[r].y, vp.x, fmaf(wi[r].x, vp.y, m.y))));
          if (row(r) == lane + 32 * q) m.y = 0.f;
          A[r][q] = m;
          if (q == Q1) first[r] = m;
          acc[2 * r] = fmaf(m.x, v.x, fmaf(-m.y, v.y, acc[2 * r]));
          acc[2 * r + 1] = fmaf(m.x, v.y, fmaf(m.y, v.x, acc[2 * r + 1]));
        }
      }
      // w' = tau A v of row r in the lanes of group r, A_{i,k+1} beside it; one lane publishes them
      const float mine = tri_sum_many<2 * NR>(acc, lane);
      const float other = __shfl_xor_sync(0xffffffffu, mine, GL / 2);
      const int rr = lane / GL, la = (k + 1) & 31;
      float2 fa = make_float2(0.f, 0.f);
#pragma unroll
      for (int r = R1; r < NR; ++r) {
        const float fx = __shfl_sync(0xffffffffu, first[r].x, la), fy = __shfl_sync(0xffffffffu, first[r].y, la);
        if (r == rr) fa = make_float2(fx, fy);
      }
      if (lane % GL == 0 && rr >= R1) {
        const float2 w = tri_mul(sh.tau[k], make_float2(mine, other));
        sh.g[b ^ 1][warp + rr * NWARP] = make_float4(w.x, w.y, fa.x, fa.y);
      }
      barrier();
    }
    if constexpr (Q1 + 1 < Q) {
      if (n - 1 > 32 * Q1 + 31) slot_steps<Q1 + 1>();
    }
  }

  // The whole reduction: load(i, j) is element (i, j) of the matrix for i, j < n.  Call with all threads.
  template <class Load> __device__ __forceinline__ void run(const Load& load) {
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int i = row(r), j = lane + 32 * q;
        A[r][q] = i < n && j < n ? load(i, j) : make_float2(0.f, 0.f);
        if (i == j) A[r][q].y = 0.f;
      }
    for (int i = threadIdx.x; i < MAXN; i += THREADS) sh.v[0][i] = sh.v[1][i] = sh.w[i] = make_float2(0.f, 0.f);
    if (lane == 0)
#pragma unroll
      for (int r = 0; r < NR; ++r) sh.g[0][warp + r * NWARP] = make_float4(0.f, 0.f, A[r][0].x, A[r][0].y);
#pragma unroll
    for (int q = 0; q < Q; ++q) vp0[q] = make_float2(0.f, 0.f);
    tk = make_float2(0.f, 0.f);
    barrier();
    slot_steps<0>();
    if (rank == 0) {
      const int j = n - 1;
      if (warp == 0 && lane == (j & 31)) {
        const float4 q = gsrc[(j & 1) * ML + j / CL];
        float dl = q.z;
        if (n >= 2) {
          // last pending update (v_{n-2} = (1))
          const float2 h = tri_mul(tk, make_float2(q.x, -q.y));
          dl -= 2.f * (q.x - 0.5f * h.x);
        }
        sh.d[j] = dl;
        sh.e[j] = 0.f;
        sh.tau[j] = make_float2(0.f, 0.f);
      }
      if (warp == 1 && n >= 2) store_reflector(n - 2, sh.v[(n - 2) & 1]);
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += THREADS) {
        T.d[i] = sh.d[i];
        T.e[i] = sh.e[i];
        T.tau[i] = sh.tau[i];
      }
    }
    barrier();                                                       // no CTA leaves while it is read
  }
};

}  // namespace ks
