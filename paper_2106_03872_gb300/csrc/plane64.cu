// FP64 transforms between the packed sphere and the full grid [x][y][z], for the grids whose (y, z) plane
// of complex128 fits an SM's shared memory (N <= 96 of the compiled sizes):
//   k_p64_inv  one x-plane of one state per CTA: the packed coefficients in, inverse z and y transforms
//   k_p64_x    16 consecutive z of one y per CTA: the x lines, only the planes that hold columns read
//              (inverse) or written (forward)
//   k_p64_fwd  forward y and z transforms of an x-plane, then scale u + |G|^2/2 c on the sphere
// The FP64 pipe bounds them (two lanes a clock per SM: the transforms of an H application of 8 states on
// 24^3 take 22 us of it); as six passes through HBM with run-time lengths they took 15, 15 and 10 us a
// pass there, the whole H application 88 us; with these it takes 78 us.
//
// Only the planes that hold columns are launched, 2 xr + 1 of N: with the others' CTAs in the grid, which
// left at once, the scheduler put two planes on some multiprocessors and none on others (3 states on 54^3
// 275 -> 208 us an H application, 6 states on 36^3 160 -> 115 us).
#include "fft_device.cuh"
#include "kernels.h"

namespace ks {

namespace {

template <int N> struct P64 {
  static constexpr int PT = N <= 36 ? 192 : 256;
  static constexpr int LPC = N <= 36 ? N : 32;                       // lines per call
  static constexpr int LB = 16;                                      // z of an x-line block (256-byte rows)
  static constexpr size_t SMEM = (size_t)(N + N * (N + 1)) * sizeof(double2);
  static constexpr size_t XSMEM = (size_t)(N + LB * (N + 1)) * sizeof(double2);
};

__device__ __forceinline__ bool in_band(int x, int N, int xr) { return x <= xr || x >= N - xr; }
// The p-th x-plane that holds columns, p < 2 xr + 1; the others are zero and the x lines do not read them.
__device__ __forceinline__ int band_plane(int p, int N, int xr) { return p <= xr ? p : N - (2 * xr + 1) + p; }

template <int N>
__global__ void __launch_bounds__(P64<N>::PT)
    k_p64_inv(const double2* __restrict__ psi, int nG, const int* __restrict__ ginv, int xr, double2* __restrict__ grid,
              const double2* __restrict__ twg) {
  constexpr int ld = N + 1, PT = P64<N>::PT;
  extern __shared__ __align__(16) double2 p64sm[];
  chain_begin();
  double2 *tw = p64sm, *P = p64sm + N;                               // [y][z]
  const int x = band_plane(blockIdx.x, N, xr), b = blockIdx.y;
  for (int t = threadIdx.x; t < N; t += PT) tw[t] = twg[t];
  const int* gi = ginv + x * N * N;
  for (int e = threadIdx.x; e < N * N; e += PT) {
    const int g = gi[e];
    P[(e / N) * ld + e % N] = g >= 0 ? psi[(size_t)b * nG + g] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  cfft_lines<N, PT, P64<N>::LPC, true, +1>(P, N, ld, 1, tw);
  cfft_lines<N, PT, P64<N>::LPC, true, +1>(P, N, 1, ld, tw);
  double2* out = grid + ((size_t)b * N + x) * N * N;
  for (int e = threadIdx.x; e < N * N; e += PT) out[e] = P[(e / N) * ld + e % N];
}

template <int N, int SIGN>
__global__ void __launch_bounds__(P64<N>::PT)
    k_p64_x(double2* __restrict__ grid, int xr, const double2* __restrict__ twg) {
  constexpr int ld = N + 1, PT = P64<N>::PT, LB = P64<N>::LB;
  extern __shared__ __align__(16) double2 p64sm[];
  chain_begin();
  double2 *tw = p64sm, *s = p64sm + N;                               // [z - z0][x]
  const int z0 = blockIdx.x * LB, y = blockIdx.y, nl = min(LB, N - z0);
  double2* at = grid + (size_t)blockIdx.z * N * N * N + (size_t)y * N + z0;
  for (int t = threadIdx.x; t < N; t += PT) tw[t] = twg[t];
  for (int e = threadIdx.x; e < N * LB; e += PT) {
    const int x = e / LB, l = e % LB;
    if (l < nl)
      s[l * ld + x] = SIGN < 0 || in_band(x, N, xr) ? at[(size_t)x * N * N + l] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  cfft_lines<N, PT, LB, true, SIGN>(s, nl, ld, 1, tw);
  for (int e = threadIdx.x; e < N * LB; e += PT) {
    const int x = e / LB, l = e % LB;
    if (l < nl && (SIGN > 0 || in_band(x, N, xr))) at[(size_t)x * N * N + l] = s[l * ld + x];
  }
}

template <int N>
__global__ void __launch_bounds__(P64<N>::PT)
    k_p64_fwd(const double2* __restrict__ grid, const double2* __restrict__ psi, double2* __restrict__ hpsi, int nG,
              const int* __restrict__ ginv, const double* __restrict__ g2h, int xr, double scale,
              const double2* __restrict__ twg) {
  constexpr int ld = N + 1, PT = P64<N>::PT;
  extern __shared__ __align__(16) double2 p64sm[];
  chain_begin();
  double2 *tw = p64sm, *P = p64sm + N;                               // [y][z]
  const int x = band_plane(blockIdx.x, N, xr), b = blockIdx.y;
  for (int t = threadIdx.x; t < N; t += PT) tw[t] = twg[t];
  const double2* in = grid + ((size_t)b * N + x) * N * N;
  for (int e = threadIdx.x; e < N * N; e += PT) P[(e / N) * ld + e % N] = in[e];
  __syncthreads();
  cfft_lines<N, PT, P64<N>::LPC, true, -1>(P, N, 1, ld, tw);
  cfft_lines<N, PT, P64<N>::LPC, true, -1>(P, N, ld, 1, tw);
  const int* gi = ginv + x * N * N;
  for (int e = threadIdx.x; e < N * N; e += PT) {
    const int g = gi[e];
    if (g < 0) continue;
    const size_t i = (size_t)b * nG + g;
    const double2 u = P[(e / N) * ld + e % N], c = psi[i];
    const double k = g2h[g];
    hpsi[i] = make_double2(u.x * scale + k * c.x, u.y * scale + k * c.y);
  }
}

// Whether nb states go through planes.  Their launch fills the GPU in steps of one plane an SM; where it
// leaves most of the last step empty, the line passes, which spread evenly, are faster: they win from
// LINES times as many plane slots as the nb N planes of the whole grids (us of an H application, planes and
// lines: 150 and 94 for 1 state on 48^3, slots 3.2 times the planes; 174 and 134 for 1 on 54^3, 2.8; 163 and
// 127 for 1 on 64^3, 2.4; 279 and 252 for 1 on 72^3, 2.1, and 507 and 450 for 3 with 61 planes each, 1.41;
// level for 2 on 36^3, 2.1; but 186 and 235 for 2 on 54^3, 1.41, and 352 and 372 for 1 on 96^3, 1.58).  Up to
// 32 points the launches count, two less with planes.
constexpr int SMS = 152;
template <int N> bool planes_pay(int nb, int xr) {
  constexpr double LINES = N == 72 ? 1.4 : 2.2;
  const long planes = (long)nb * (2 * xr + 1), slots = (planes + SMS - 1) / SMS * SMS;
  return N <= 32 || slots <= LINES * nb * N;
}

// The element count that decides on a chained launch (launch_chain) of the forward passes.  Where mid-sized
// work leaves SMs idle, the planes of the last pass, set up early, pile up on them and then run several to
// an SM while the others have none: 3 us of launch latency hidden, up to 70 us lost (H application of 2
// states on 72^3 374 us chained, 300 not; 6 on 36^3 147 and 111; 2 on 64^3 220 and 178).  Chained: the
// smallest work (24^3, 4 states: 57 and 68 us), grids from 48 points on whose planes fill the SMs (64^3, 4
// states: 288 and 300), and 96 points, whose planes take an SM's whole shared memory (1 state: 338 and 352).
// The inverse passes are level at every size and always chained.
template <int N> size_t chain_elems(int nb, int xr) {
  const size_t pts = (size_t)nb * N * N * N;
  const bool chain = pts <= (size_t(1) << 17) || N >= 96 || (N >= 48 && (long)nb * (2 * xr + 1) >= SMS);
  return chain ? pts : CHAIN_ELEMS + 1;
}

template <int N> struct NTag {
  static constexpr int value = N;
};
template <typename F> bool with_planes(int N, int nb, int xr, F&& f) {
  auto go = [&](auto tag) {
    if (!planes_pay<decltype(tag)::value>(nb, xr)) return false;
    f(tag);
    return true;
  };
  switch (N) {
    case 24: return go(NTag<24>{});
    case 32: return go(NTag<32>{});
    case 36: return go(NTag<36>{});
    case 48: return go(NTag<48>{});
    case 54: return go(NTag<54>{});
    case 64: return go(NTag<64>{});
    case 72: return go(NTag<72>{});
    case 96: return go(NTag<96>{});
    default: return false;
  }
}

}  // namespace

bool plane64_inverse(const double2* psi, double2* grid, const int* ginv, const DevTables<double>& t, int nb,
                     cudaStream_t s) {
  return with_planes(t.N, nb, t.xr, [&](auto tag) {
    constexpr int N = decltype(tag)::value;
    static bool attr = false;
    if (!attr) {
      KS_CUDA(cudaFuncSetAttribute(k_p64_inv<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P64<N>::SMEM));
      attr = true;
    }
    const size_t pts = (size_t)nb * N * N * N;
    launch_chain(pts, k_p64_inv<N>, dim3(2 * t.xr + 1, nb), dim3(P64<N>::PT), P64<N>::SMEM, s, psi, t.nG, ginv,
                 t.xr, grid, t.tw);
    launch_chain(pts, k_p64_x<N, +1>, dim3((N + P64<N>::LB - 1) / P64<N>::LB, N, nb), dim3(P64<N>::PT), P64<N>::XSMEM, s,
                 grid, t.xr, t.tw);
  });
}

bool plane64_forward(double2* grid, const double2* psi, double2* hpsi, const int* ginv, const DevTables<double>& t,
                     int nb, double scale, cudaStream_t s) {
  return with_planes(t.N, nb, t.xr, [&](auto tag) {
    constexpr int N = decltype(tag)::value;
    static bool attr = false;
    if (!attr) {
      KS_CUDA(cudaFuncSetAttribute(k_p64_fwd<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P64<N>::SMEM));
      attr = true;
    }
    const size_t pts = chain_elems<N>(nb, t.xr);
    launch_chain(pts, k_p64_x<N, -1>, dim3((N + P64<N>::LB - 1) / P64<N>::LB, N, nb), dim3(P64<N>::PT), P64<N>::XSMEM, s,
                 grid, t.xr, t.tw);
    launch_chain(pts, k_p64_fwd<N>, dim3(2 * t.xr + 1, nb), dim3(P64<N>::PT), P64<N>::SMEM, s, grid, psi, hpsi, t.nG,
                 ginv, t.g2half, t.xr, scale, t.tw);
  });
}

}  // namespace ks
