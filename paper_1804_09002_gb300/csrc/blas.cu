// Dense FP64 building blocks: batched/grouped GEMM on the FP64 FMA pipe,
// elementwise kernels and deterministic reductions.
//
// GB300 executes FP64 at about 2 DFMA per clock per SM (the f64 mma.sync path
// is slower still), so these kernels are bound by the DFMA pipe, not by HBM:
// the GEMM keeps a 4x4 register tile per thread fed from shared memory, which
// needs one shared-memory load per two FMAs, and relies on several resident
// CTAs per SM to cover global-load latency.  Grids are sized by the output
// tiles of all problems of a batch together.
#include <type_traits>

#include "ops.h"
#include "tc_gemm.h"

namespace zcsd {

namespace {

constexpr int NT = 256;

// Output tile BM x BN, RM x RN outputs per thread (256 threads), k-step BK.
// The next k-step's operands are loaded into registers before the current
// one is consumed (not where a thread's complex 4 x 4 outputs fill them).
// Tiles of fewer than 256 outputs share every k-step among KG groups of
// threads, whose sums are added at the end.  A warp instruction holds its
// scheduler's FP64 lanes for 64 clocks, so nothing is issued that can be left
// out: unit weights and alpha, rows and columns beyond the edge.
template <class T, int OPA, int OPB, int BM, int BN, int RM, int RN, int BK>
__global__ void __launch_bounds__(NT, 2) gemm_kernel(GemmArgs<T> g) {
  constexpr int TX = BM / RM, TY = BN / RN;  // thread grid over the tile
  constexpr int KG = NT / (TX * TY);
  static_assert(TX * TY * KG == NT && TX * TY % 32 == 0 && BK % KG == 0, "256 threads, whole warps per group");
  constexpr int LA = BM * BK / NT, LB = BN * BK / NT;
  constexpr bool AHEAD = sizeof(T) == 8 || RM * RN < 16;
  const int z = blockIdx.z;
  const int b = z / g.ksplit, ks = z % g.ksplit;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  chain_wait();
  if (g.uplo == 1 && m0 > n0 + BN - 1) return;
  if (g.uplo == 2 && n0 > m0 + BM - 1) return;
  int kb = 0, ke = g.k;
  if (g.ksplit > 1) {
    const int kc = ((g.k + g.ksplit - 1) / g.ksplit + 15) / 16 * 16;
    kb = ks * kc;
    ke = min(g.k, kb + kc);
  }
  if (g.kflags & K_FROM_COL) kb = max(kb, n0);
  if (g.kflags & K_FROM_ROW) kb = max(kb, m0);
  if (g.kflags & K_TO_COL) ke = min(ke, n0 + BN);
  if (g.kflags & K_TO_ROW) ke = min(ke, m0 + BM);

  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid % (TX * TY) / TX, kg = tid / (TX * TY);
  // outputs inside the matrix: row blocks of the tile, column blocks of the warp
  const int rows = min(RM, (g.m - m0 + TX - 1) / TX);
  const int cols = min(RN, (g.n - n0 - (tid & ~31) % (TX * TY) / TX + TY - 1) / TY);
  T acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = zero<T>();

  T va[LA], vb[LB];
  const int k00 = (kb / 16) * 16, steps = ke > k00 ? (ke - k00 + BK - 1) / BK : 0;
  // ---- op(A)[m0:m0+BM, kt:kt+BK] and op(B)[kt:kt+BK, n0:n0+BN] into
  // registers, coalesced along memory
  auto fetch = [&](int it) {
    const int js = it / steps, kt = k00 + (it % steps) * BK;
    const T* A = g.A + (b / g.bdivA) * g.sA + js * g.sAj;
    const T* B = g.B + (b / g.bdivB) * g.sB + js * g.sBj;
    const double wj = g.w[js];
#pragma unroll
    for (int s = 0; s < LA; ++s) {
      const int e = tid + NT * s;
      const int i = (OPA == OP_N) ? (e % BM) : (e / BK);
      const int k = (OPA == OP_N) ? (e / BM) : (e % BK);
      const int gi = m0 + i, gk = kt + k;
      T v = zero<T>();
      if (gi < g.m && gk >= kb && gk < ke) {
        if (OPA == OP_N) v = A[gi + (long long)gk * g.lda];
        else {
          v = A[gk + (long long)gi * g.lda];
          if (OPA == OP_C) v = conj_(v);
        }
      }
      va[s] = wj != 1.0 ? scal(wj, v) : v;
    }
#pragma unroll
    for (int s = 0; s < LB; ++s) {
      const int e = tid + NT * s;
      const int k = (OPB == OP_N) ? (e % BK) : (e / BN);
      const int j = (OPB == OP_N) ? (e / BK) : (e % BN);
      const int gj = n0 + j, gk = kt + k;
      T v = zero<T>();
      if (gj < g.n && gk >= kb && gk < ke) {
        if (OPB == OP_N) v = B[gk + (long long)gj * g.ldb];
        else {
          v = B[gj + (long long)gk * g.ldb];
          if (OPB == OP_C) v = conj_(v);
        }
      }
      vb[s] = v;
    }
  };
  const int total = steps * g.nsum;
  if (AHEAD && total > 0) fetch(0);
  for (int it = 0; it < total; ++it) {
    if (!AHEAD) fetch(it);
#pragma unroll
    for (int s = 0; s < LA; ++s) {
      const int e = tid + NT * s;
      As[(OPA == OP_N) ? (e / BM) : (e % BK)][(OPA == OP_N) ? (e % BM) : (e / BK)] = va[s];
    }
#pragma unroll
    for (int s = 0; s < LB; ++s) {
      const int e = tid + NT * s;
      Bs[(OPB == OP_N) ? (e % BK) : (e / BN)][(OPB == OP_N) ? (e / BK) : (e % BN)] = vb[s];
    }
    __syncthreads();
    if (AHEAD && it + 1 < total) fetch(it + 1);
#pragma unroll
    for (int kk = 0; kk < BK; kk += KG) {
      const int k = kk + kg;
      T a[RM], bb[RN];
#pragma unroll
      for (int i = 0; i < RM; ++i) a[i] = As[k][tx + TX * i];
#pragma unroll
      for (int j = 0; j < RN; ++j) bb[j] = Bs[k][ty + TY * j];
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j)
          if (i < rows && j < cols) acc[i][j] = fmac(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }
  if constexpr (KG > 1) {
    static_assert(RM == 1 && RN == 1 && (KG - 1) * BM * BN <= BK * (BM + 1), "sums of the groups fit As");
    T* sums = &As[0][0];
    if (kg > 0) sums[tid - BM * BN] = acc[0][0];
    __syncthreads();
    if (kg > 0) return;
#pragma unroll
    for (int s = 0; s < KG - 1; ++s) acc[0][0] = add(acc[0][0], sums[tid + s * BM * BN]);
  }
  // ---- epilogue
  chain_next();
  T* C = g.C + z * g.sC;
  const T* Cin = g.Cin ? g.Cin + (b / g.bdivC) * g.sCin : nullptr;
  const bool unit = re(g.alpha) == 1.0 && im(g.alpha) == 0.0;
  const bool use_beta = Cin && ks == 0 && (re(g.beta) != 0.0 || im(g.beta) != 0.0);
#pragma unroll
  for (int j = 0; j < RN; ++j) {
    const int gj = n0 + ty + TY * j;
    if (gj >= g.n) continue;
#pragma unroll
    for (int i = 0; i < RM; ++i) {
      const int gi = m0 + tx + TX * i;
      if (gi >= g.m) continue;
      T v = unit ? acc[i][j] : mul(g.alpha, acc[i][j]);
      if (use_beta) v = fmac(g.beta, Cin[gi + (long long)gj * g.ldcin], v);
      C[gi + (long long)gj * g.ldc] = v;
    }
  }
}

// Tiles of the FP64 product.  The pipe (two multiply-adds per clock and SM) is
// the bound at every tile size, one output per thread included, so the tile
// is the one whose fullest SM has the least to do: ceil(tiles / 152) tiles of
// BM x BN outputs.  128^3 (two problems): 64 x 64 tiles on 8 SMs take 130 us,
// 16 x 16 tiles 9 us.  Large outputs keep 64 x 64 (32 x 128 for m <= 32),
// which read each operand least often; a smaller tile has to win by 10 %.
// The products between the 32-column blocks of an inverse Cholesky factor fill
// the chip with 8 x 8 tiles only (csd n = 64 1.65 -> 1.53 ms, n = 201 6.60 ->
// 6.13, polar n = 2048 42.8 -> 41.1, together with what the kernel leaves out).
// A product in place needs one tile over the whole of what it overwrites, and
// the column tiles must fit a grid's second dimension (more than 524 280 columns
// are too many for 8-column tiles).
enum GemmTile { TILE_64 = 0, TILE_32x128, TILE_32, TILE_16, TILE_16x8, TILE_8, TILES };
constexpr int TILE_M[TILES] = {64, 32, 32, 16, 16, 8}, TILE_N[TILES] = {64, 128, 32, 16, 8, 8};

template <class T>
int pick_tile(const GemmArgs<T>& g) {
  int best = -1;
  double cost = 0.0;
  for (int t = 0; t < TILES; ++t) {
    if ((g.C == g.B && TILE_M[t] < g.m) || (g.C == g.A && TILE_N[t] < g.n)) continue;
    if (ceil_div(g.n, TILE_N[t]) > 65535) continue;
    const long long tm = ceil_div(g.m, TILE_M[t]), tn = ceil_div(g.n, TILE_N[t]);
    long long tiles = tm * tn;
    if (g.uplo) tiles = (tiles + std::min(tm, tn)) / 2;
    tiles *= (long long)g.batch * g.ksplit;
    const double c = (double)ceil_div(tiles, 152) * TILE_M[t] * TILE_N[t];
    if (best < 0 || c < 0.9 * cost) {
      best = t;
      cost = c;
    }
  }
  return best < 0 ? TILE_64 : best;
}

template <class T, int OPA, int OPB>
void gemm_launch(const GemmArgs<T>& g, int tile, cudaStream_t st) {
  const dim3 grid(ceil_div(g.m, TILE_M[tile]), ceil_div(g.n, TILE_N[tile]), g.batch * g.ksplit);
  switch (tile) {
    case TILE_64: launch_chained(gemm_kernel<T, OPA, OPB, 64, 64, 4, 4, 16>, grid, NT, 0, st, g); break;
    case TILE_32x128: launch_chained(gemm_kernel<T, OPA, OPB, 32, 128, 4, 4, 16>, grid, NT, 0, st, g); break;
    case TILE_32: launch_chained(gemm_kernel<T, OPA, OPB, 32, 32, 2, 2, 16>, grid, NT, 0, st, g); break;
    case TILE_16: launch_chained(gemm_kernel<T, OPA, OPB, 16, 16, 1, 1, 32>, grid, NT, 0, st, g); break;
    case TILE_16x8: launch_chained(gemm_kernel<T, OPA, OPB, 16, 8, 1, 1, 32>, grid, NT, 0, st, g); break;
    default: launch_chained(gemm_kernel<T, OPA, OPB, 8, 8, 1, 1, 32>, grid, NT, 0, st, g); break;
  }
}

template <class T, int OPA>
void gemm_dispatch_b(const GemmArgs<T>& g, int tile, cudaStream_t st) {
  if (g.opB == OP_N) gemm_launch<T, OPA, OP_N>(g, tile, st);
  else if (g.opB == OP_C && sizeof(T) == 16) gemm_launch<T, OPA, OP_C>(g, tile, st);
  else gemm_launch<T, OPA, OP_T>(g, tile, st);
}

template <class T>
void gemm_dispatch(const GemmArgs<T>& g, int tile, cudaStream_t st) {
  if (g.opA == OP_N) gemm_dispatch_b<T, OP_N>(g, tile, st);
  else if (g.opA == OP_C && sizeof(T) == 16) gemm_dispatch_b<T, OP_C>(g, tile, st);
  else gemm_dispatch_b<T, OP_T>(g, tile, st);
}

// Multiply-add work the kernel executes for g, counted per output tile over
// the k range it traverses (2 flops per real FMA, 8 per complex FMA).
template <class T>
double gemm_flops(const GemmArgs<T>& g, int BM, int BN) {
  double fma = 0.0;
  const int tm = ceil_div(g.m, BM), tn = ceil_div(g.n, BN);
  for (int bx = 0; bx < tm; ++bx) {
    const int m0 = bx * BM, rows = std::min(BM, g.m - m0);
    for (int by = 0; by < tn; ++by) {
      const int n0 = by * BN, cols = std::min(BN, g.n - n0);
      if (g.uplo == 1 && m0 > n0 + BN - 1) continue;
      if (g.uplo == 2 && n0 > m0 + BM - 1) continue;
      int kb = 0, ke = g.k;
      if (g.kflags & K_FROM_COL) kb = std::max(kb, n0);
      if (g.kflags & K_FROM_ROW) kb = std::max(kb, m0);
      if (g.kflags & K_TO_COL) ke = std::min(ke, n0 + BN);
      if (g.kflags & K_TO_ROW) ke = std::min(ke, m0 + BM);
      if (ke > kb) fma += (double)rows * cols * (ke - kb);
    }
  }
  return fma * g.nsum * g.batch * (sizeof(T) == sizeof(double) ? 2.0 : 8.0);
}

}  // namespace

template <class T>
void gemm(const GemmArgs<T>& g, cudaStream_t st) {
  if (g.m <= 0 || g.n <= 0 || g.batch <= 0) return;
  if constexpr (std::is_same<T, double>::value) {
    if (tc_will_handle(g)) {
      tc_gemm(g, st, *t_tc.ar, t_tc.err);
      return;
    }
  } else {
    if (tc_will_handle_complex(g)) {
      tc_gemm_complex(g, st, *t_tc.ar, t_tc.err);
      return;
    }
  }
  ProfToken tok = prof_begin(st);
  const int tile = pick_tile(g);
  gemm_dispatch<T>(g, tile, st);
  ZCSD_LAUNCH();
  if (tok.slot >= 0) prof_end(tok, st, PK_GEMM, gemm_flops(g, TILE_M[tile], TILE_N[tile]), g.site);
}

template <class T>
void gemm1(cudaStream_t st, int opA, int opB, int m, int n, int k, T alpha, const T* A, int lda,
           const T* B, int ldb, T beta, T* C, int ldc, int uplo, int kflags, int site) {
  GemmArgs<T> g;
  g.site = site;
  g.m = m; g.n = n; g.k = k; g.opA = opA; g.opB = opB;
  g.A = A; g.lda = lda; g.B = B; g.ldb = ldb;
  g.Cin = C; g.ldcin = ldc; g.C = C; g.ldc = ldc;
  g.alpha = alpha; g.beta = beta; g.uplo = uplo; g.kflags = kflags;
  gemm(g, st);
}

// ------------------------------------------------------------------ elementwise
namespace {

struct Vec16 {
  double v[MAX_SUM];
};

template <class F>
__global__ void ew2d_kernel(int m, int n, int batch, F f) {
  const long long total = (long long)m * n;
  const int b = blockIdx.y;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % m), j = (int)(t / m);
    f(i, j, b);
  }
  (void)batch;
}

template <class F>
void ew2d(cudaStream_t st, int m, int n, int batch, F f) {
  if (m <= 0 || n <= 0 || batch <= 0) return;
  long long total = (long long)m * n;
  int blocks = (int)std::min<long long>((total + 255) / 256, 152 * 8);
  ew2d_kernel<<<dim3(blocks, batch), 256, 0, st>>>(m, n, batch, f);
  ZCSD_LAUNCH();
}

}  // namespace

template <class T>
void axpby(cudaStream_t st, int m, int n, double alpha, const T* X, int ldx, long long sX, double beta, T* Y,
           int ldy, long long sY, int batch) {
  ew2d(st, m, n, batch, [=] __device__(int i, int j, int b) {
    T x = scal(alpha, X[b * sX + i + (long long)j * ldx]);
    T* y = Y + b * sY + i + (long long)j * ldy;
    *y = (beta != 0.0) ? add(x, scal(beta, *y)) : x;
  });
}

template <class T>
void sum_parts(cudaStream_t st, int m, int n, T* X, int ldx, long long sPart, int parts, int batch) {
  if (parts <= 1) return;
  ew2d(st, m, n, batch, [=] __device__(int i, int j, int b) {
    T* x = X + (long long)b * parts * sPart + i + (long long)j * ldx;
    T acc = *x;
    for (int s = 1; s < parts; ++s) acc = add(acc, x[s * sPart]);
    *x = acc;
  });
}

template <class T>
void shift_terms(cudaStream_t st, int n, const T* X, int ldx, long long sXb, const double* shifts, int nterms,
                 T* Y, int ldy, long long sY, int batch) {
  Vec16 s;
  for (int j = 0; j < MAX_SUM; ++j) s.v[j] = j < nterms ? shifts[j] : 0.0;
  // problem index p = b * nterms + jterm
  ew2d(st, n, n, batch * nterms, [=] __device__(int i, int j, int p) {
    const int bb = p / nterms, jt = p % nterms;
    T x = X[bb * sXb + i + (long long)j * ldx];
    if (i == j) x = add(x, from_re<T>(s.v[jt]));
    Y[p * sY + i + (long long)j * ldy] = x;
  });
}

template <class T>
void stack_terms(cudaStream_t st, int n, const T* X, int ldx, long long sXb, const double* sqrtc, int nterms,
                 T* M, int ldm, long long sM, int batch) {
  Vec16 s;
  for (int j = 0; j < MAX_SUM; ++j) s.v[j] = j < nterms ? sqrtc[j] : 0.0;
  ew2d(st, 2 * n, n, batch * nterms, [=] __device__(int i, int j, int p) {
    const int bb = p / nterms, jt = p % nterms;
    T v;
    if (i < n) v = X[bb * sXb + i + (long long)j * ldx];
    else v = (i - n == j) ? from_re<T>(s.v[jt]) : zero<T>();
    M[p * sM + i + (long long)j * ldm] = v;
  });
}

template <class T>
void scale_shift(cudaStream_t st, int n, double alpha, const T* X, int ldx, long long sX, double beta, T* Z, int ldz,
                 long long sZ, int batch) {
  ew2d(st, n, n, batch, [=] __device__(int i, int j, int b) {
    T x = scal(alpha, X[b * sX + i + (long long)j * ldx]);
    if (i == j) x = add(x, from_re<T>(beta));
    Z[b * sZ + i + (long long)j * ldz] = x;
  });
}

template <class T>
void scale_terms(cudaStream_t st, int m, int n, const double* s_, int nterms, T* X, int ldx, long long sX, int batch) {
  Vec16 s;
  for (int j = 0; j < MAX_SUM; ++j) s.v[j] = j < nterms ? s_[j] : 0.0;
  ew2d(st, m, n, batch * nterms, [=] __device__(int i, int j, int p) {
    T* x = X + p * sX + i + (long long)j * ldx;
    *x = scal(s.v[p % nterms], *x);
  });
}

template <class T>
void minus_eye(cudaStream_t st, int n, const T* X, int ldx, long long sX, T* E, int lde, long long sE, int batch) {
  ew2d(st, n, n, batch, [=] __device__(int i, int j, int b) {
    if (i > j) return;
    T x = X[b * sX + i + (long long)j * ldx];
    if (i == j) x = from_re<T>(re(x) - 1.0);
    E[b * sE + i + (long long)j * lde] = x;
    if (i < j) E[b * sE + j + (long long)i * lde] = conj_(x);
  });
}

template <class T>
void mirror(cudaStream_t st, int n, T* X, int ldx, long long sX, int batch) {
  ew2d(st, n, n, batch, [=] __device__(int i, int j, int b) {
    if (i < j) X[b * sX + j + (long long)i * ldx] = conj_(X[b * sX + i + (long long)j * ldx]);
  });
}

template <class T>
void symmetrize(cudaStream_t st, int n, const T* Y, int ldy, long long sY, T* H, int ldh, long long sH, int batch) {
  // each (i, j) with i <= j handled once, so in-place use is race-free
  ew2d(st, n, n, batch, [=] __device__(int i, int j, int b) {
    if (i > j) return;
    const T a = Y[b * sY + i + (long long)j * ldy];
    const T c = Y[b * sY + j + (long long)i * ldy];
    const T h = scal(0.5, add(a, conj_(c)));
    H[b * sH + i + (long long)j * ldh] = h;
    H[b * sH + j + (long long)i * ldh] = conj_(h);
    if (i == j) H[b * sH + i + (long long)i * ldh] = from_re<T>(re(h));
  });
}

template <class T>
void set_eye(cudaStream_t st, int m, int n, T* E, int lde, long long sE, int batch) {
  ew2d(st, m, n, batch, [=] __device__(int i, int j, int b) {
    E[b * sE + i + (long long)j * lde] = (i == j) ? from_re<T>(1.0) : zero<T>();
  });
}

// ------------------------------------------------------------------ reductions
namespace {

constexpr int RED_BLOCKS = 304;  // 2 per SM; partial sums are combined in fixed order

__device__ inline double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
  }
  __syncthreads();
  return r;
}

template <class T>
__global__ void fro2_partial(int m, int n, const T* X, int ldx, long long sX, double shift, double* part) {
  __shared__ double sh[32];
  const int b = blockIdx.y;
  const long long total = (long long)m * n;
  double acc = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % m), j = (int)(t / m);
    T x = X[b * sX + i + (long long)j * ldx];
    if (i == j) x = sub(x, from_re<T>(shift));
    acc += abs2(x);
  }
  const double r = block_sum(acc, sh);
  if (threadIdx.x == 0) part[b * gridDim.x + blockIdx.x] = r;
}

__global__ void finish_sum(const double* part, int nparts, int batch, double* out) {
  __shared__ double sh[32];
  for (int b = 0; b < batch; ++b) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += part[b * nparts + i];
    const double r = block_sum(acc, sh);
    if (threadIdx.x == 0) out[b] = r;
  }
}

template <class T>
__global__ void nonfinite_partial(int m, int n, const T* X, int ldx, double* part) {
  __shared__ double sh[32];
  const long long total = (long long)m * n;
  double acc = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % m), j = (int)(t / m);
    const T x = X[i + (long long)j * ldx];
    if (!isfinite(re(x)) || !isfinite(im(x))) acc += 1.0;
  }
  const double r = block_sum(acc, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = r;
}

template <class T>
__global__ void col_dots_kernel(int m, int n, const T* V, int ldv, const T* Y, int ldy, double* d) {
  __shared__ double sh[32];
  const int j = blockIdx.x;
  double acc = 0.0;
  for (int i = threadIdx.x; i < m; i += blockDim.x)
    acc += re(cmul(V[i + (long long)j * ldv], Y[i + (long long)j * ldy]));
  const double r = block_sum(acc, sh);
  if (threadIdx.x == 0) d[j] = r;
}

template <class T>
__global__ void diag_real_kernel(int n, const T* X, int ldx, double* d) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    d[i] = re(X[i + (long long)i * ldx]);
}

// theta = atan2(S, C) clamped to [0, pi/2], the range of the principal
// angles (Section 1); rounding can otherwise leave S or C a few ulps below 0.
// v clamped to [lo, hi]; NaN stays NaN (fmin and fmax would hide a failed factor)
__device__ inline double clamp_keep_nan(double v, double lo, double hi) { return v <= lo ? lo : (v > hi ? hi : v); }

__global__ void theta_kernel(int n, const double* C, const double* S, double* th) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    th[i] = clamp_keep_nan(atan2(S[i], C[i]), 0.0, 1.5707963267948966);
}

// remark (iv): theta solves sin(theta) - cos(theta) = Lambda, i.e.
// sqrt(2) sin(theta - pi/4) = Lambda, theta = pi/4 + asin(Lambda / sqrt(2)),
// with Lambda / sqrt(2) clamped to [-1, 1] and theta to [0, pi/2].
__global__ void theta_lambda_kernel(int n, const double* lam, double* th) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double x = clamp_keep_nan(lam[i] * 0.70710678118654752, -1.0, 1.0);
    th[i] = clamp_keep_nan(0.78539816339744831 + asin(x), 0.0, 1.5707963267948966);
  }
}

// rank of each key among all keys (ties by index): perm[rank] = index, a warp
// per key.  NaN keys order after +inf, so the ranks always form a permutation.
// A thread per key compared on the FP64 pipe of n / 256 SMs: 303 us at n =
// 1024.
__global__ void __launch_bounds__(256) sort_perm_kernel(int n, const double* key, int* perm) {
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  const int r = warp_rank(key, n, i);
  if ((threadIdx.x & 31) == 0) perm[r] = i;
}

template <class T>
__global__ void gather_cols_kernel(int m, int ncols, const T* X, int ldx, const int* perm, T* Y, int ldy) {
  const long long total = (long long)m * ncols;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % m), j = (int)(t / m);
    const int pj = perm[j];
    // perm is a permutation of [0, ncols); the guard only keeps a corrupted
    // index from reading outside X
    Y[i + (long long)j * ldy] = (pj >= 0 && pj < ncols) ? X[i + (long long)pj * ldx] : from_re<T>(NAN);
  }
}

__global__ void gather_vec_kernel(int n, const double* x, const int* perm, double* y) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int p = perm[i];
    y[i] = (p >= 0 && p < n) ? x[p] : NAN;
  }
}

// splitmix64 (Steele, Lea and Flood 2014): a bijective 64-bit mixer used as a
// counter-based generator, stream position = element index.
__device__ inline unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ inline double unit_open(unsigned long long r) {  // (0, 1)
  return ((double)(r >> 11) + 0.5) * 0x1p-53;
}

template <class T>
__global__ void randn_kernel(int m, int n, T* X, int ldx, unsigned long long seed) {
  const long long total = (long long)m * n;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % m), j = (int)(t / m);
    const unsigned long long base = seed * 0x100000001B3ull + (unsigned long long)t * 2ull;
    const double u1 = unit_open(splitmix64(base)), u2 = unit_open(splitmix64(base + 1));
    const double rad = sqrt(-2.0 * log(u1));
    double s, c;
    sincospi(2.0 * u2, &s, &c);
    T v;
    if constexpr (sizeof(T) == sizeof(double)) v = from_re<T>(rad * c);
    else { z64 z{rad * c * 0.7071067811865476, rad * s * 0.7071067811865476}; v = *reinterpret_cast<T*>(&z); }
    X[i + (long long)j * ldx] = v;
  }
}

}  // namespace

template <class T>
void fro2(cudaStream_t st, int m, int n, const T* X, int ldx, long long sX, double shift, double* out, int batch,
          double* scratch) {
  if (m <= 0 || n <= 0) {
    ZCSD_CUDA(cudaMemsetAsync(out, 0, sizeof(double) * batch, st));
    return;
  }
  fro2_partial<T><<<dim3(RED_BLOCKS, batch), 256, 0, st>>>(m, n, X, ldx, sX, shift, scratch);
  ZCSD_LAUNCH();
  finish_sum<<<1, 256, 0, st>>>(scratch, RED_BLOCKS, batch, out);
  ZCSD_LAUNCH();
}

template <class T>
void count_nonfinite(cudaStream_t st, int m, int n, const T* X, int ldx, double* out, double* scratch) {
  nonfinite_partial<T><<<RED_BLOCKS, 256, 0, st>>>(m, n, X, ldx, scratch);
  ZCSD_LAUNCH();
  finish_sum<<<1, 256, 0, st>>>(scratch, RED_BLOCKS, 1, out);
  ZCSD_LAUNCH();
}

template <class T>
void col_dots(cudaStream_t st, int m, int n, const T* V, int ldv, const T* Y, int ldy, double* d) {
  if (n <= 0) return;
  col_dots_kernel<T><<<n, 256, 0, st>>>(m, n, V, ldv, Y, ldy, d);
  ZCSD_LAUNCH();
}

template <class T>
void diag_real(cudaStream_t st, int n, const T* X, int ldx, double* d) {
  if (n <= 0) return;
  diag_real_kernel<T><<<ceil_div(n, 256), 256, 0, st>>>(n, X, ldx, d);
  ZCSD_LAUNCH();
}

void theta_from_cs(cudaStream_t st, int n, const double* C, const double* S, double* theta) {
  if (n <= 0) return;
  theta_kernel<<<ceil_div(n, 256), 256, 0, st>>>(n, C, S, theta);
  ZCSD_LAUNCH();
}

void theta_from_lambda(cudaStream_t st, int n, const double* lam, double* theta) {
  if (n <= 0) return;
  theta_lambda_kernel<<<ceil_div(n, 256), 256, 0, st>>>(n, lam, theta);
  ZCSD_LAUNCH();
}

void sort_perm(cudaStream_t st, int n, const double* key, int* perm) {
  if (n <= 0) return;
  sort_perm_kernel<<<ceil_div(n, 8), 256, 0, st>>>(n, key, perm);
  ZCSD_LAUNCH();
}

template <class T>
void gather_cols(cudaStream_t st, int m, int ncols, const T* X, int ldx, const int* perm, T* Y, int ldy) {
  if (m <= 0 || ncols <= 0) return;
  long long total = (long long)m * ncols;
  gather_cols_kernel<T><<<(int)std::min<long long>((total + 255) / 256, 152 * 8), 256, 0, st>>>(m, ncols, X, ldx,
                                                                                              perm, Y, ldy);
  ZCSD_LAUNCH();
}

void gather_vec(cudaStream_t st, int n, const double* x, const int* perm, double* y) {
  if (n <= 0) return;
  gather_vec_kernel<<<ceil_div(n, 256), 256, 0, st>>>(n, x, perm, y);
  ZCSD_LAUNCH();
}

template <class T>
void randn(cudaStream_t st, int m, int n, T* X, int ldx, unsigned long long seed) {
  long long total = (long long)m * n;
  if (total <= 0) return;
  randn_kernel<T><<<(int)std::min<long long>((total + 255) / 256, 152 * 8), 256, 0, st>>>(m, n, X, ldx, seed);
  ZCSD_LAUNCH();
}

// ------------------------------------------------------------------ instantiations
#define ZCSD_INST(T)                                                                                             \
  template void gemm<T>(const GemmArgs<T>&, cudaStream_t);                                                      \
  template void gemm1<T>(cudaStream_t, int, int, int, int, int, T, const T*, int, const T*, int, T, T*, int, int, \
                         int, int);                                                                                \
  template void axpby<T>(cudaStream_t, int, int, double, const T*, int, long long, double, T*, int, long long, int); \
  template void sum_parts<T>(cudaStream_t, int, int, T*, int, long long, int, int);                                  \
  template void shift_terms<T>(cudaStream_t, int, const T*, int, long long, const double*, int, T*, int, long long, \
                               int);                                                                            \
  template void stack_terms<T>(cudaStream_t, int, const T*, int, long long, const double*, int, T*, int, long long, \
                               int);                                                                            \
  template void scale_shift<T>(cudaStream_t, int, double, const T*, int, long long, double, T*, int, long long, int); \
  template void scale_terms<T>(cudaStream_t, int, int, const double*, int, T*, int, long long, int);            \
  template void minus_eye<T>(cudaStream_t, int, const T*, int, long long, T*, int, long long, int);             \
  template void mirror<T>(cudaStream_t, int, T*, int, long long, int);                                          \
  template void symmetrize<T>(cudaStream_t, int, const T*, int, long long, T*, int, long long, int);            \
  template void set_eye<T>(cudaStream_t, int, int, T*, int, long long, int);                                    \
  template void fro2<T>(cudaStream_t, int, int, const T*, int, long long, double, double*, int, double*);       \
  template void count_nonfinite<T>(cudaStream_t, int, int, const T*, int, double*, double*);                    \
  template void col_dots<T>(cudaStream_t, int, int, const T*, int, const T*, int, double*);                     \
  template void diag_real<T>(cudaStream_t, int, const T*, int, double*);                                        \
  template void gather_cols<T>(cudaStream_t, int, int, const T*, int, const int*, T*, int);                     \
  template void randn<T>(cudaStream_t, int, int, T*, int, unsigned long long);

ZCSD_INST(double)
ZCSD_INST(z64)

}  // namespace zcsd
