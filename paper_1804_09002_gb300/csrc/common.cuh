// Shared device/host definitions of the Zolo-csd CUDA library.
//
// Matrices are column-major with an explicit leading dimension, FP64 real
// (double) or complex (z64 = {re, im}).  All kernels are templated on the
// scalar type T through the small set of helpers below.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstdio>

namespace zcsd {

struct z64 {
  double x, y;
};

// ---------------------------------------------------------------- scalars
__host__ __device__ inline double re(double a) { return a; }
__host__ __device__ inline double re(z64 a) { return a.x; }
__host__ __device__ inline double im(double) { return 0.0; }
__host__ __device__ inline double im(z64 a) { return a.y; }
__host__ __device__ inline double conj_(double a) { return a; }
__host__ __device__ inline z64 conj_(z64 a) { return {a.x, -a.y}; }
__host__ __device__ inline double abs2(double a) { return a * a; }
__host__ __device__ inline double abs2(z64 a) { return a.x * a.x + a.y * a.y; }
template <class T> __host__ __device__ inline T from_re(double a);
template <> __host__ __device__ inline double from_re<double>(double a) { return a; }
template <> __host__ __device__ inline z64 from_re<z64>(double a) { return {a, 0.0}; }
template <class T> __host__ __device__ inline T zero() { return from_re<T>(0.0); }
__host__ __device__ inline double add(double a, double b) { return a + b; }
__host__ __device__ inline z64 add(z64 a, z64 b) { return {a.x + b.x, a.y + b.y}; }
__host__ __device__ inline double sub(double a, double b) { return a - b; }
__host__ __device__ inline z64 sub(z64 a, z64 b) { return {a.x - b.x, a.y - b.y}; }
__host__ __device__ inline double mul(double a, double b) { return a * b; }
__host__ __device__ inline z64 mul(z64 a, z64 b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
__host__ __device__ inline double scal(double s, double a) { return s * a; }
__host__ __device__ inline z64 scal(double s, z64 a) { return {s * a.x, s * a.y}; }
// c + a*b
__host__ __device__ inline double fmac(double a, double b, double c) { return fma(a, b, c); }
__host__ __device__ inline z64 fmac(z64 a, z64 b, z64 c) {
  return {fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y))};
}
// conj(a)*b
__host__ __device__ inline double cmul(double a, double b) { return a * b; }
__host__ __device__ inline z64 cmul(z64 a, z64 b) {
  return {a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x};
}
__host__ __device__ inline double div_(double a, double b) { return a / b; }
__host__ __device__ inline z64 div_(z64 a, z64 b) {
  double d = b.x * b.x + b.y * b.y;
  return {(a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d};
}

template <class T> struct dtype_id;
template <> struct dtype_id<double> { static constexpr int value = 0; };
template <> struct dtype_id<z64> { static constexpr int value = 1; };

// ---------------------------------------------------------------- ranks
#ifdef __CUDACC__
// 64-bit integers in the order of the doubles, -0 equal to +0 and every NaN
// after +inf: an integer comparison costs a fraction of one on the FP64 pipe.
__device__ inline long long order_key(double v) {
  const long long b = __double_as_longlong(v), mag = b & 0x7FFFFFFFFFFFFFFFll;
  if (mag > 0x7FF0000000000000ll) return 0x7FFFFFFFFFFFFFFFll;
  return b >= 0 ? b : -mag;
}

// rank of x[i] among x[0 .. n), ties by index, by one warp (the same value in
// every lane)
__device__ inline int warp_rank(const double* x, int n, int i) {
  const long long v = order_key(x[i]);
  int r = 0;
  for (int k = threadIdx.x & 31; k < n; k += 32) {
    const long long w = order_key(x[k]);
    r += w < v || (w == v && k < i);
  }
  return (int)__reduce_add_sync(0xffffffffu, (unsigned)r);
}
#endif

// ---------------------------------------------------------------- errors
// Library-internal error carrier: a CUDA error is turned into a status code
// at the C-ABI boundary.
struct CudaFail {
  cudaError_t err;
  const char* file;
  int line;
};

#define ZCSD_CUDA(call)                                     \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) throw ::zcsd::CudaFail{e_, __FILE__, __LINE__}; \
  } while (0)

// Every kernel launch goes through ZCSD_LAUNCH(), which also counts it.
void count_launch();
#define ZCSD_LAUNCH()                  \
  do {                                 \
    ::zcsd::count_launch();            \
    ZCSD_CUDA(cudaGetLastError());     \
  } while (0)

#ifdef __CUDACC__
// Kernels of the long chains of short launches (small products, Cholesky
// blocks, Jacobi rounds) are launched while their predecessor ends: every
// thread that touches memory first waits for all of the predecessor
// (chain_wait), and a CTA that has only its results left to write lets the
// successor's CTAs in (chain_next; a CTA that exits counts too).  A kernel
// launched without the attribute waits as ever, and so does whatever follows a
// chained kernel without it.  csd n = 64 1.50 -> 1.37 ms, n = 500 14.5 -> 12.9,
// n = 1024 38.9 -> 35.5, polar n = 2048 41.2 -> 38.3.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
void launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ZCSD_CUDA(cudaLaunchKernelEx(&cfg, kernel, P(args)...));
}
#endif

// Optional per-kind kernel timing (CUDA events on the launch stream), used
// for roofline reports.  prof_begin/prof_end bracket one launch; both are
// no-ops unless a profiler is active on the calling thread.
enum ProfKind { PK_GEMM = 0, PK_QR_PANEL = 1, PK_POTRF = 2, PK_JACOBI = 3, PK_TC = 4, PK_KINDS = 5 };
struct ProfToken {
  int slot = -1;
};
ProfToken prof_begin(cudaStream_t st);
void prof_end(ProfToken t, cudaStream_t st, int kind, double flops, int site = 0);
constexpr int PROF_SITES = 24;

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

}  // namespace zcsd
