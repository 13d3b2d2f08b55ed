// Shared host/device definitions of the CUDA path: error handling, complex types,
// the host geometry tables.  Nothing here is shared with the oracle.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <string>
#include <vector>

#include "ks.h"

namespace ks {

// ---------------------------------------------------------------------------------------------
// Errors: internal code throws ks::Error; every ABI entry point catches it and returns st.
// ---------------------------------------------------------------------------------------------
struct Error {
  ks_status st;
};

void set_last_error(const std::string& msg);
[[noreturn]] void fail(ks_status st, const char* fmt, ...);
[[noreturn]] void fail_cuda(cudaError_t e, const char* what, const char* file, int line);

#define KS_CUDA(call)                                                  \
  do {                                                                 \
    cudaError_t e_ = (call);                                           \
    if (e_ != cudaSuccess) ks::fail_cuda(e_, #call, __FILE__, __LINE__); \
  } while (0)

// Every kernel launch is followed by KS_CHECK_LAUNCH(): it counts the launch (reported by
// ks_kernel_launches) and turns a launch error into ks::Error.
void note_launch();
#define KS_CHECK_LAUNCH()          \
  do {                             \
    ks::note_launch();             \
    KS_CUDA(cudaGetLastError());   \
  } while (0)

// Chained launches: a kernel launched with launch_chain may be set up while the kernel before it on the
// stream still runs (programmatic stream serialization); it calls chain_begin() before anything else,
// which waits until everything before it on the stream has completed, so the order of the work is the
// stream's.  What it hides is the launch latency between dependent kernels, 2 to 4 us each: of the six
// kernels of 3 to 8 us in an H application of a small cell, half the time (24^3, 8 states: 36 -> 23 us; 20
// real-time steps of 24 states on 32^3: 9.95 -> 7.4 ms).
// `elems`, the values the kernel works on, decides: above CHAIN_ELEMS the kernel runs long enough to
// hide its successor's launch by itself, and being set up early harms it: its blocks pile up on the
// multiprocessors that the kernel before it leaves first (512 states on 128^3, a step: 96.3 ms without,
// 103.8 ms with every launch chained; 64 states on 64^3, 1.7e7 points, an SCF call: 4.41 ms without,
// 4.20 ms with).
constexpr size_t CHAIN_ELEMS = size_t(1) << 25;
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
void launch_chain(size_t elems, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = elems <= CHAIN_ELEMS ? 1 : 0;
  KS_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
  KS_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------------------------
// Complex types: float2 / double2 with the few operations the kernels use.
// ---------------------------------------------------------------------------------------------
template <typename T> struct cplx_of;
template <> struct cplx_of<float> { using type = float2; };
template <> struct cplx_of<double> { using type = double2; };
template <typename T> using cplx = typename cplx_of<T>::type;

template <typename C> __host__ __device__ __forceinline__ C mk(decltype(C::x) r, decltype(C::x) i) {
  C c;
  c.x = r;
  c.y = i;
  return c;
}
// On the device the sums, differences and products of complex64 values are packed pairs (add, mul and
// fma on two FP32 values of one 64-bit register pair, the same roundings): half the instructions of the
// butterflies, which are what the FFT kernels issue most.  Plane kernel per H application of 128^3 states
// 51.4 -> 49.9 ms (8 x 512 states), of 64^3 118 -> 114 us (64 states); at 96 points the packing costs the
// registers it saves in instructions (0.616 and 0.620 ms).
__device__ __forceinline__ unsigned long long f2_bits(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 f2_of(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__host__ __device__ __forceinline__ float2 operator+(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ float2 operator-(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  const float2 m = make_float2(-1.f, -1.f);
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(b)), "l"(f2_bits(m)), "l"(f2_bits(a)));
  return f2_of(r);
#else
  return make_float2(a.x - b.x, a.y - b.y);
#endif
}
__host__ __device__ __forceinline__ float2 operator*(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__host__ __device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ double2 operator*(double2 a, double s) { return make_double2(a.x * s, a.y * s); }

template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
#ifdef __CUDA_ARCH__
  if constexpr (sizeof(C) == 8) {
    unsigned long long t, r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(f2_bits(make_float2(-a.y, a.x))), "l"(f2_bits(make_float2(b.y, b.y))));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(make_float2(a.x, a.y))), "l"(f2_bits(make_float2(b.x, b.x))), "l"(t));
    return f2_of(r);
  }
#endif
  return mk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// conj(a) * b
template <typename C> __host__ __device__ __forceinline__ C cmulc(C a, C b) {
  return mk<C>(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

// ---------------------------------------------------------------------------------------------
// Host geometry: cutoff sphere, z-columns, V_loc, projector spheres (built once per handle).
// ---------------------------------------------------------------------------------------------
struct HostGeometry {
  double L = 0, h = 0, omega = 0, dV = 0, ecut = 0;
  int N = 0, nG = 0;
  std::vector<int> gidx;        // packed G -> flat grid index (jx*N + jy)*N + jz
  std::vector<int> mvec;        // [nG][3] integer frequencies
  std::vector<double> g2half;   // |G|^2 / 2
  // z-columns of the sphere: a column (jx, jy) holds cnt = 2*hz+1 consecutive packed
  // entries; entry k sits at jz = k (k <= hz) or jz = N - cnt + k (k > hz).
  int ncols = 0;
  std::vector<int> col_xy;      // jx*N + jy, increasing
  std::vector<int> col_off;     // first packed index of the column
  std::vector<int> col_half;    // hz
  int xr = 0;                   // columns exist only for |m_x| <= xr (and |m_y| <= xr)
  double vmin = 0, vmax = 0;     // extremes of V_loc (formed on the device)
  std::vector<double> pos;      // [natoms][3] atom positions (bohr)
  double vloc_depth = 0, vloc_width = 0;
  // projectors: sphere point lists per atom (grid order within an atom)
  int natoms = 0, nproj = 0;
  double D = 0, proj_sigma = 0, proj_rc = 0;
  std::vector<int> sph_off;     // [natoms+1]
  std::vector<int> sph_idx;     // flat grid index of each sphere point
  std::vector<int> sph_atom;    // atom of each sphere point
  std::vector<double> sph_beta; // [npts][nproj]
  std::vector<int> sph_zorder;  // [npts] the atom's sphere points visited plane by plane (z, then x, y)
  // inverse lists: every grid point covered by >= 1 sphere, with its sphere points in atom order
  std::vector<int> cov_idx;     // flat grid index, increasing
  std::vector<int> cov_off;     // [ncov+1]
  std::vector<int> cov_ent;     // sphere point indices
  std::vector<int> cov_scratch; // [N^3 + 1] counts, kept between rebuilds (no page faults per move)
  std::vector<double> occ;      // [nstates]
  std::vector<double> tw;       // [N][2] cos, sin of 2 pi t / N
};

bool valid_fft_length(int N);
void count_sphere(double L, int N, double ecut, int* nG);
void build_geometry(const ks_cell_desc& d, HostGeometry& g);
// Rebuilds the atom-dependent parts (pos, the projector sphere lists and their inverse lists)
// for new positions pos [natoms][3] of the same atoms.  V_loc, vmin and vmax are the
// engine's to fill (on the device).
void build_atoms(const double* pos, HostGeometry& g);
// Grid steps from its centre beyond which a Gaussian of this width is below 1e-20 (at most N).
int gaussian_half_box(double width, double h, int N);

}  // namespace ks
