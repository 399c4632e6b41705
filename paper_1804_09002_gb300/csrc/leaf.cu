// Eigendecomposition of the leaf blocks of Zolo-eig (and of every B of a
// batch), all leaves of any sizes in the same launches.  GB300 retires two
// FP64 multiply-adds per clock and SM against 128 in FP32, so an FP64 Jacobi
// sweep of a 256-row leaf is bound by that pipe and by a launch per
// tournament round.  The leaf is therefore solved in three stages:
//
//  1. FP32 one-sided Jacobi (Hestenes) on the shifted, scaled copy
//     (B - m I) / ||B - m I||_F + s I, which is positive definite, so its
//     rotated columns W = A V tend to v_j times an eigenvalue: only W is
//     stored, no eigenvector matrix and no row rotations.
//  2. FP64 refinement of X = W / ||w_j|| (Ogita and Aishima, "Iterative
//     refinement for symmetric eigenvalue decomposition", Japan J. Indust.
//     Appl. Math. 35, 2018): S = X^* B X, P = X^* X, lambda_j = s_jj / p_jj,
//     E_ij = (s_ij - lambda_j p_ij) / (lambda_j - lambda_i), X <- X + X E.
//     Each step squares the error and is three products; a pair closer than
//     four times the coupling of its columns is only re-orthogonalised.
//     Leaves that end with such clusters repeat stages 1 and 2 on them: every
//     cluster's block of S, shifted and scaled by itself, is a new FP32
//     problem at the same place (blocks of different clusters have exactly
//     orthogonal columns, so one solve serves all).  A pass resolves gaps about
//     1e-3 of its clusters' width, so spectra graded over FP64's range (small
//     angles) take up to six (n = 1000, lambda = 2^(-40 i / n): 65 ms; left to
//     stage 3 after three passes, 8.0 s).
//  3. Leaves that still hold an off-diagonal entry above rounding level are
//     finished by FP64 two-sided Jacobi on S, a cluster of CTAs per leaf, one
//     launch (on B itself, should X not be orthonormal).
//
// The accuracy is that of stages 2 and 3 alone, FP64 similarity transforms of
// B itself; stage 1 only supplies the starting basis.
//
// Measured on GB300 against cyclic FP64 Jacobi with two launches per round
// (heig of a random matrix): n = 64 6.3 -> 0.8 ms, 200 31 -> 2.1 ms; complex
// n = 512 9.4 ms.  At n = 1024 one leaf takes 16 ms (41 ms without tensor
// cores) where splitting down to 256 rows took 125 ms, hence the leaf size.
// Stage 1 is then 70 % of the time, bound by the issue slots of the few SMs
// that hold a leaf; the refinement's products run at 60 % of the FP64 pipe.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "solver.h"
#include "tc_gemm.h"

namespace cg = cooperative_groups;

namespace zcsd {

namespace {

constexpr int J32_SWEEPS = 12;          // FP32 sweeps at most
constexpr float J32_ROT = 5e-7f;        // rotate above this cosine (FP32 dot products resolve ~1e-7)
constexpr float J32_STOP = 1e-3f;       // a sweep that saw no larger cosine is the last (quadratic convergence)
constexpr int PRE_PARTS = 32, POW_STEPS = 7;
constexpr int J32_SMEM = 200 * 1024;    // columns of a block pair
constexpr int REF_STEPS = 7;            // refinement steps of a pass at most, ...
constexpr int ORTHO_STEPS = 2;          // ... the last of them only re-orthogonalise
constexpr int PASSES = 8;               // passes of stages 1 and 2 at most (later ones on clusters)
constexpr double GAP = 4.0;             // pairs closer than this many couplings are not rotated but clustered
constexpr int OFF_N = PASSES * (REF_STEPS + 1);  // looks at a leaf's state
constexpr unsigned LEAF_OPEN = 1, LEAF_SKEW = 2;  // off-diagonal above rounding; X not orthonormal
constexpr int LEAF_TC = 384;            // rows from which tensor-core products pay
constexpr int JAC_CTAS = 8;             // CTAs per leaf of the FP64 stage (portable cluster size)
constexpr int JAC_THREADS = 256;

// Column blocks of the FP32 stage of an n-row leaf: nblk (even) blocks of wb
// columns; a CTA holds two of them in shared memory.  Blocks of 32 columns
// keep n / 64 SMs busy per leaf with one launch per 32 local rounds; from 257
// floats per column on 16 columns are faster (twice the SMs, one column per
// warp and round).  Leaves of at most 96 rows are one pair
// of blocks: a single CTA, which then runs every sweep in one launch.  Across
// the blocks a warp keeps j32_owned columns of the first one in registers, so
// a block has at most j32_cover columns whatever the leaf's size (beside a leaf
// of 257 floats per column and more, a leaf of 33 to 96 rows has several pairs
// of 16 columns, which cost nothing next to that leaf's rounds).
__host__ __device__ constexpr int j32_threads(int lds) { return lds <= 256 ? 1024 : 512; }
__host__ __device__ constexpr int j32_owned(int lds) { return lds >= 384 ? 1 : 2; }
__host__ __device__ constexpr int j32_cover(int lds) { return j32_owned(lds) * j32_threads(lds) / 32; }

struct J32Geom {
  int nf;    // floats per column (n, complex 2n)
  int ldg;   // floats per stored column, a multiple of 4
  int nblk, wb;
};

__host__ __device__ inline J32Geom j32_geom(int n, bool cplx, int lds) {
  J32Geom g;
  g.nf = cplx ? 2 * n : n;
  g.ldg = (g.nf + 3) & ~3;
  int wmax = J32_SMEM / (8 * lds);
  const int cap = lds >= 384 ? 16 : 32;
  wmax = wmax > cap ? cap : wmax;
  if (n <= 96 && lds <= 512) wmax = (n + 1) / 2;
  wmax = wmax > j32_cover(lds) ? j32_cover(lds) : wmax;
  const int half = (n + 2 * wmax - 1) / (2 * wmax);
  g.nblk = 2 * (half < 1 ? 1 : half);
  g.wb = (n + g.nblk - 1) / g.nblk;
  return g;
}

// Disjoint pair k of round r in the tournament of an even number of players.
__device__ __forceinline__ void tournament(int players, int r, int k, int& p, int& q) {
  if (k == 0) {
    p = players - 1;
    q = r;
  } else {
    p = (r + k) % (players - 1);
    q = (r - k + (players - 1)) % (players - 1);
  }
  if (p > q) {
    const int x = p;
    p = q;
    q = x;
  }
}

// leaf l ended at or before look `it` (its later entries stay 0)
__device__ __forceinline__ bool leaf_ended(const LeafDev& L, int l, int it) {
  return it >= 0 && L.off[l * OFF_N + it] == 0u;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// sum over the CTA, the same value for every thread (sh: 33 doubles)
__device__ inline double cta_sum(double v, double* sh) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    double x = l < (int)(blockDim.x >> 5) ? sh[l] : 0.0;
    x = warp_sum(x);
    if (l == 0) sh[32] = x;
  }
  __syncthreads();
  const double r = sh[32];
  __syncthreads();
  return r;
}

// Partial sums of ||B_l||_F^2 and ||B_l - m I||_F^2, m = tr(B_l) / n, in a
// fixed order (blockIdx.x of PRE_PARTS); the leaf's state is cleared.
template <class T>
__global__ void __launch_bounds__(256) leaf_norm_kernel(LeafDev L, const T* B) {
  __shared__ double sh[33];
  const int l = blockIdx.y, n = L.sz[l], ld = L.ldb[l], tid = threadIdx.x;
  const T* Bl = B + L.boff[l];
  double tr = 0.0, a = 0.0, a0 = 0.0;
  for (int i = tid; i < n; i += blockDim.x) tr += re(Bl[i + (long long)i * ld]);
  const double m = cta_sum(tr, sh) / n;
  for (int t = blockIdx.x * blockDim.x + tid; t < n * n; t += PRE_PARTS * blockDim.x) {
    const int i = t % n, j = t / n;
    T v = Bl[i + (long long)j * ld];
    a += abs2(v);
    if (i == j) v = sub(v, from_re<T>(m));
    a0 += abs2(v);
  }
  a = cta_sum(a, sh);
  a0 = cta_sum(a0, sh);
  if (tid == 0) {
    L.part[(l * PRE_PARTS + blockIdx.x) * 2] = a;
    L.part[(l * PRE_PARTS + blockIdx.x) * 2 + 1] = a0;
  }
  if (blockIdx.x == 0) {
    for (int t = tid; t < OFF_N; t += blockDim.x) L.off[l * OFF_N + t] = 0u;
    for (int t = tid; t < PASSES * J32_SWEEPS; t += blockDim.x) L.cosmax[l * PASSES * J32_SWEEPS + t] = 0;
    for (int t = tid; t < JAC_SWEEPS_MAX; t += blockDim.x) L.rot[l * JAC_SWEEPS_MAX + t] = 0;
    if (tid == 0) {
      L.norms[2 * l] = m;
      L.done[l] = 0;
    }
  }
}

// W_l = (B_l - m I) / ||B_l - m I||_F in FP32; c_l = ||B_l||_F; the start
// vector of the power iteration.
template <class T>
__global__ void __launch_bounds__(256) leaf_fill_kernel(LeafDev L, const T* B, int lds) {
  constexpr bool CX = sizeof(T) == 16;
  const int l = blockIdx.y, n = L.sz[l], ld = L.ldb[l];
  const T* Bl = B + L.boff[l];
  double a = 0.0, a0 = 0.0;
  for (int k = 0; k < PRE_PARTS; ++k) {
    a += L.part[(l * PRE_PARTS + k) * 2];
    a0 += L.part[(l * PRE_PARTS + k) * 2 + 1];
  }
  const double m = L.norms[2 * l], inv = a0 > 0.0 ? 1.0 / sqrt(a0) : 0.0;
  const J32Geom g = j32_geom(n, CX, lds);
  float* W = L.w32 + L.woff[l];
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < g.ldg * n; t += gridDim.x * blockDim.x) {
    const int f = t % g.ldg, j = t / g.ldg, i = CX ? f >> 1 : f;
    float w = 0.0f;
    if (i < n) {
      const T v = Bl[i + (long long)j * ld];
      if (i == j) w = (CX && (f & 1)) ? 0.0f : (float)((re(v) - m) * inv);
      else w = (float)(((CX && (f & 1)) ? im(v) : re(v)) * inv);
    }
    W[t] = w;
  }
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      L.c[l] = a > 0.0 ? sqrt(a) : 1.0;
      L.norms[2 * l + 1] = sqrt(a0);
    }
    for (int i = threadIdx.x; i < g.nf; i += blockDim.x) {
      unsigned h = (unsigned)i * 2654435761u + 12345u;  // a fixed vector without structure
      h ^= h >> 15;
      h *= 2246822519u;
      h ^= h >> 13;
      L.x32[4 * L.voff[l] + i] = (float)(int)h * 4.656613e-10f;
    }
  }
}

// Step `it` of the power iteration, y = W x / ||x|| (W Hermitian: one warp per
// column); step POW_STEPS instead adds s = 1.3 ||x|| to the diagonal.  The
// scaled matrix's 2-norm is at most 1; an estimate that is too small costs
// only the separation of lambda and -lambda - 2 s, which the later stages
// repair.
template <bool CX>
__global__ void __launch_bounds__(256) leaf_power_kernel(LeafDev L, int it, int lds) {
  __shared__ double sh[33];
  const int l = blockIdx.y, n = L.sz[l], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blockIdx.x * 8 >= n) return;
  const J32Geom g = j32_geom(n, CX, lds);
  const float* x = L.x32 + 4 * L.voff[l] + (it & 1) * g.nf;
  float* y = L.x32 + 4 * L.voff[l] + ((it + 1) & 1) * g.nf;
  double nx = 0.0;
  for (int i = threadIdx.x; i < g.nf; i += blockDim.x) nx += (double)(x[i] * x[i]);
  const float r = (float)sqrt(cta_sum(nx, sh));
  const int j = blockIdx.x * 8 + warp;
  if (j >= n) return;
  float* w = L.w32 + L.woff[l] + (long long)j * g.ldg;
  if (it == POW_STEPS) {
    const float s = r > 0.0f ? 1.3f * r : 1.0f;
    if (lane == 0) {
      w[CX ? 2 * j : j] += s;
      // about ||B_l||_2, the scale of the rounding errors of S
      if (j == 0) L.norms[2 * l + 1] = fmin(L.c[l], fabs(L.norms[2 * l]) + L.norms[2 * l + 1] * (double)s);
    }
    return;
  }
  const float sc = r > 0.0f ? 1.0f / r : 0.0f;
  float sr = 0.0f, si = 0.0f;
  for (int i = lane; i < n; i += 32) {
    if (CX) {
      const float wr = w[2 * i], wi = w[2 * i + 1], xr = x[2 * i], xi = x[2 * i + 1];
      sr += wr * xr + wi * xi;
      si += wr * xi - wi * xr;
    } else {
      sr += w[i] * x[i];
    }
  }
  sr = warp_sum(sr);
  if (CX) si = warp_sum(si);
  if (lane == 0) {
    if (CX) {
      y[2 * j] = sr * sc;
      y[2 * j + 1] = si * sc;
    } else {
      y[j] = sr * sc;
    }
  }
}

// One round of the block tournament: a CTA loads two column blocks of its
// leaf (NV float4 per lane and column), rotates every pair across them (and,
// in round 0, every pair inside each) and writes them back.  One warp per
// column pair: the dot product by shuffles, both columns in registers from
// the product to the rotation, column norms kept in shared memory.
template <bool CX, int NV, int THREADS>
__global__ void __launch_bounds__(THREADS) j32_kernel(LeafDev L, int pass, int sweep, int round) {
  extern __shared__ __align__(16) float j32_smem[];
  __shared__ float nrm[96];
  __shared__ int cmax;
  constexpr int LDS = 128 * NV, NW = THREADS / 32;
  chain_wait();
  const int l = blockIdx.y, n = L.sz[l];
  const J32Geom g = j32_geom(n, CX, LDS);
  if ((int)blockIdx.x >= g.nblk / 2 || round >= g.nblk - 1) return;
  const bool whole = g.nblk == 2;  // this CTA holds the leaf: all sweeps in the first launch
  if (whole && sweep > 0) return;
  if (leaf_ended(L, l, pass * (REF_STEPS + 1) - 1)) return;
  int* cosmax = L.cosmax + (l * PASSES + pass) * J32_SWEEPS;
  if (sweep > 0 && __int_as_float(cosmax[sweep - 1]) < J32_STOP * J32_STOP) return;
  int bp, bq;
  tournament(g.nblk, round, blockIdx.x, bp, bq);
  const int wb = g.wb, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* W = L.w32 + L.woff[l];
  float4* S4 = reinterpret_cast<float4*>(j32_smem);
  for (int c = warp; c < 2 * wb; c += NW) {
    const int col = (c < wb ? bp * wb + c : bq * wb + c - wb);
    const bool on = col < n && col < (c < wb ? bp + 1 : bq + 1) * wb;
    const float4* src = reinterpret_cast<const float4*>(W + (long long)col * g.ldg);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int e = v * 32 + lane;
      float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      if (on && 4 * e < g.ldg) z = src[e];
      S4[c * (LDS / 4) + e] = z;
    }
  }
  if (tid == 0) cmax = 0;
  __syncthreads();

  float seen = 0.0f;  // largest squared cosine this warp met in the sweep
  auto norms = [&]() {
    for (int c = warp; c < 2 * wb; c += NW) {
      float a = 0.0f;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float4 z = S4[c * (LDS / 4) + v * 32 + lane];
        a += z.x * z.x + z.y * z.y + z.z * z.z + z.w * z.w;
      }
      a = warp_sum(a);
      if (lane == 0) nrm[c] = a;
    }
  };
  auto load = [&](int c, float4 (&z)[NV]) {
#pragma unroll
    for (int v = 0; v < NV; ++v) z[v] = S4[c * (LDS / 4) + v * 32 + lane];
  };
  auto store = [&](int c, const float4 (&z)[NV]) {
#pragma unroll
    for (int v = 0; v < NV; ++v) S4[c * (LDS / 4) + v * 32 + lane] = z[v];
  };
  // rotates columns x and y (squared norms al, be); false: nothing to do.
  // The phase of g = x^* y moves into y, tan 2 phi = 2 |g| / (be - al).
  // Approximate reciprocals and roots: their 1e-7 is the columns' rounding.
  auto rotate = [&](float4 (&x)[NV], float4 (&y)[NV], float& al, float& be) -> bool {
    if (!(al > 0.0f && be > 0.0f)) return false;
    float gr = 0.0f, gi = 0.0f;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      gr += x[v].x * y[v].x + x[v].y * y[v].y + x[v].z * y[v].z + x[v].w * y[v].w;
      if (CX) gi += x[v].x * y[v].y - x[v].y * y[v].x + x[v].z * y[v].w - x[v].w * y[v].z;
    }
    gr = warp_sum(gr);
    if (CX) gi = warp_sum(gi);
    const float g2 = CX ? gr * gr + gi * gi : gr * gr;
    const float cos2 = __fdividef(g2, al * be);
    seen = fmaxf(seen, cos2);
    if (!(cos2 > J32_ROT * J32_ROT)) return false;
    const float ig = rsqrtf(g2), gm = g2 * ig;
    const float pr = CX ? gr * ig : copysignf(1.0f, gr), pi = CX ? gi * ig : 0.0f;
    const float zeta = 0.5f * (be - al) * ig, az = fminf(fabsf(zeta), 1e9f);
    const float w = 1.0f + az * az;
    const float t = copysignf(__fdividef(1.0f, az + w * rsqrtf(w)), zeta);
    const float c = rsqrtf(1.0f + t * t), s = c * t;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const float4 a = x[v];
      float4 b;
      if (CX) {
        b.x = y[v].x * pr + y[v].y * pi;
        b.y = y[v].y * pr - y[v].x * pi;
        b.z = y[v].z * pr + y[v].w * pi;
        b.w = y[v].w * pr - y[v].z * pi;
      } else {
        b = y[v];
      }
      // real: the sign of g goes into the coefficients
      const float sb = CX ? s : s * pr, cb = CX ? c : c * pr;
      x[v] = make_float4(c * a.x - sb * b.x, c * a.y - sb * b.y, c * a.z - sb * b.z, c * a.w - sb * b.w);
      y[v] = make_float4(s * a.x + cb * b.x, s * a.y + cb * b.y, s * a.z + cb * b.z, s * a.w + cb * b.w);
    }
    al -= t * gm;
    be += t * gm;
    return true;
  };
  auto pair = [&](int p, int q) {
    float4 x[NV], y[NV];
    float al = nrm[p], be = nrm[q];
    load(p, x);
    load(q, y);
    if (rotate(x, y, al, be)) {
      store(p, x);
      store(q, y);
      __syncwarp();
      if (lane == 0) {
        nrm[p] = al;
        nrm[q] = be;
      }
    }
  };
  static_assert(THREADS == j32_threads(LDS), "the column blocks are sized for these warps");
  constexpr int KP = j32_owned(LDS);  // columns of the first block a warp owns across the blocks
  constexpr bool KEEP = NV <= 8;      // ... in registers
  auto cross = [&]() {
    if constexpr (KEEP) {
      float4 x[KP][NV];
      float al[KP];
#pragma unroll
      for (int a = 0; a < KP; ++a) {
        const int p = warp + a * NW;
        al[a] = 0.0f;
        if (p < wb) {
          load(p, x[a]);
          al[a] = nrm[p];
        }
      }
      for (int r = 0; r < wb; ++r) {
#pragma unroll
        for (int a = 0; a < KP; ++a) {
          const int p = warp + a * NW;
          if (p >= wb) continue;
          const int q = wb + (p + r < wb ? p + r : p + r - wb);
          float4 y[NV];
          float be = nrm[q];
          load(q, y);
          if (rotate(x[a], y, al[a], be)) {
            store(q, y);
            __syncwarp();
            if (lane == 0) nrm[q] = be;
          }
        }
        __syncthreads();
      }
#pragma unroll
      for (int a = 0; a < KP; ++a)
        if (warp + a * NW < wb) store(warp + a * NW, x[a]);
    } else {
      for (int r = 0; r < wb; ++r) {
        for (int k = warp; k < wb; k += NW) pair(k, wb + (k + r) % wb);
        __syncthreads();
      }
    }
  };

  for (int sw = whole ? 0 : sweep; sw < J32_SWEEPS; ++sw) {
    norms();
    __syncthreads();
    if (round == 0) {  // pairs inside each block, both blocks side by side
      const int wp = wb + (wb & 1), half = wp / 2;
      for (int r = 0; r < wp - 1; ++r) {
        for (int k = warp; k < 2 * half; k += NW) {
          int p, q;
          tournament(wp, r, k % half, p, q);
          const int o = k < half ? 0 : wb;
          if (q < wb) pair(o + p, o + q);
        }
        __syncthreads();
      }
    }
    cross();
    if (lane == 0) atomicMax(&cmax, __float_as_int(seen));
    seen = 0.0f;
    if (!whole) break;
    __syncthreads();
    const float worst = __int_as_float(cmax);
    __syncthreads();
    if (tid == 0) cmax = 0;
    __syncthreads();
    if (worst < J32_STOP * J32_STOP) break;
  }
  chain_next();
  for (int c = warp; c < 2 * wb; c += NW) {
    const int col = (c < wb ? bp * wb + c : bq * wb + c - wb);
    if (!(col < n && col < (c < wb ? bp + 1 : bq + 1) * wb)) continue;
    float4* dst = reinterpret_cast<float4*>(W + (long long)col * g.ldg);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int e = v * 32 + lane;
      if (4 * e < g.ldg) dst[e] = S4[c * (LDS / 4) + e];
    }
  }
  if (!whole) {
    __syncthreads();
    if (tid == 0) atomicMax(&cosmax[sweep], cmax);
  }
}

// X_l = columns of W_l scaled to norm 1 (one warp per column); a column that
// FP32 lost (zero or not finite) becomes a unit vector.
template <class T>
__global__ void leaf_basis_kernel(LeafDev L, int pass, T* X, int lds) {
  constexpr bool CX = sizeof(T) == 16;
  const int l = blockIdx.y, n = L.sz[l], lane = threadIdx.x & 31;
  if (leaf_ended(L, l, pass * (REF_STEPS + 1) - 1)) return;
  const J32Geom g = j32_geom(n, CX, lds);
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (j >= n) return;
  const float* w = L.w32 + L.woff[l] + (long long)j * g.ldg;
  double a = 0.0;
  for (int i = lane; i < g.nf; i += 32) a += (double)w[i] * (double)w[i];
  a = warp_sum(a);
  const bool ok = a > 0.0 && a < 1e300;
  const double inv = ok ? 1.0 / sqrt(a) : 0.0;
  T* x = X + L.goff[l] + (long long)j * n;
  for (int i = lane; i < n; i += 32) {
    T v;
    if constexpr (CX) v = z64{(double)w[2 * i] * inv, (double)w[2 * i + 1] * inv};
    else v = (double)w[i] * inv;
    x[i] = ok ? v : from_re<T>(i == j ? 1.0 : 0.0);
  }
}

// largest coupling |s_ij - lambda_j p_ij| that ends the refinement: a few
// times the rounding of a computed entry of S, which is of order u ||B||_2
// (rotating by what is below it would only add noise inside clusters).  For a
// spread spectrum it is about the u ||B||_F that stage 3 rotates down to.
__device__ __forceinline__ double off_tol(const LeafDev& L, int l) {
  return fmax(6.0, 0.4 * sqrt((double)L.sz[l])) * 0x1p-53 * L.norms[2 * l + 1];
}

// Products of the refinement, every leaf in one launch, 16 x 8 tiles (the
// FP64 pipe is the bound, so small tiles that spread evenly over the SMs beat
// reuse: a 200-row leaf gives 325 CTAs).
//  MM_BX: T = B X      MM_GRAM: S = X^* T and P = X^* X (z = 0, 1; upper
//  tiles, mirrored)    MM_XE: P = X + X E (E in T's buffer)
//  MM_XY: P = X Y (Y in T's buffer)
enum { MM_BX = 0, MM_GRAM = 1, MM_XE = 2, MM_XY = 3 };
constexpr int MM_R = 16, MM_C = 8, MM_K = 32;

template <class T, int MODE>
__global__ void __launch_bounds__(MM_R * MM_C) leaf_mm_kernel(LeafDev L, int it, int max_n, const T* B, T* X,
                                                              T* Tm, T* S, T* P) {
  __shared__ T sa[MM_K][MM_R + 1], sb[MM_K][MM_C + 1];
  const int l = blockIdx.y, n = L.sz[l];
  const int tr = (n + MM_R - 1) / MM_R, tc = (n + MM_C - 1) / MM_C;
  if ((int)blockIdx.x >= tr * tc || n > max_n) return;
  if (leaf_ended(L, l, MODE == MM_XE ? it : it - 1)) return;
  const int i0 = (blockIdx.x % tr) * MM_R, j0 = (blockIdx.x / tr) * MM_C;
  if (MODE == MM_GRAM && i0 > j0 + MM_C - 1) return;  // below the diagonal: written by its mirror
  const long long o = L.goff[l];
  const int ld = L.ldb[l];
  const T* A_ = MODE == MM_BX ? B + L.boff[l] : X + o;
  const T* B_ = MODE == MM_BX ? X + o : (MODE == MM_GRAM ? (blockIdx.z == 0 ? Tm + o : X + o) : Tm + o);
  const int lda = MODE == MM_BX ? ld : n;
  const int tid = threadIdx.x, ti = tid % MM_R, tj = tid / MM_R;
  T acc = zero<T>();
  for (int k0 = 0; k0 < n; k0 += MM_K) {
    for (int e = tid; e < MM_K * MM_R; e += MM_R * MM_C) {
      int i, k;
      if (MODE == MM_GRAM) {
        k = e % MM_K;
        i = e / MM_K;
      } else {
        i = e % MM_R;
        k = e / MM_R;
      }
      T v = zero<T>();
      if (i0 + i < n && k0 + k < n) {
        if (MODE == MM_GRAM) v = conj_(A_[(k0 + k) + (long long)(i0 + i) * lda]);
        else v = A_[(i0 + i) + (long long)(k0 + k) * lda];
      }
      sa[k][i] = v;
    }
    for (int e = tid; e < MM_K * MM_C; e += MM_R * MM_C) {
      const int k = e % MM_K, j = e / MM_K;
      sb[k][j] = (j0 + j < n && k0 + k < n) ? B_[(k0 + k) + (long long)(j0 + j) * n] : zero<T>();
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < MM_K; ++k) acc = fmac(sa[k][ti], sb[k][tj], acc);
    __syncthreads();
  }
  const int i = i0 + ti, j = j0 + tj;
  if (i >= n || j >= n) return;
  if (MODE == MM_BX) {
    Tm[o + i + (long long)j * n] = acc;
  } else if (MODE == MM_GRAM) {
    if (i > j) return;
    T* D = blockIdx.z == 0 ? S : P;
    if (i == j) acc = from_re<T>(re(acc));
    D[o + i + (long long)j * n] = acc;
    D[o + j + (long long)i * n] = conj_(acc);
  } else {
    P[o + i + (long long)j * n] = MODE == MM_XE ? add(X[o + i + (long long)j * n], acc) : acc;
  }
}

// Column j of a leaf (a warp): lambda_j, rho_j = ||(s_ij - lambda_j p_ij)_{i != j}||
// and the leaf's state at look `it`: 0 when every coupling and |p_ij - delta_ij|
// is at its rounding level.  A pass that ends with couplings of u ||B||_F at most
// ends the leaf as well: the FP64 stage would not rotate them, and a wide leaf's
// rounding can keep a cluster's couplings just above the other level for ever.
template <class T>
__global__ void leaf_state_kernel(LeafDev L, int it, const T* S, const T* P) {
  const int l = blockIdx.y, n = L.sz[l], lane = threadIdx.x & 31;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (j >= n || leaf_ended(L, l, it - 1)) return;
  const T* s = S + L.goff[l] + (long long)j * n;
  const T* p = P + L.goff[l] + (long long)j * n;
  const bool last = it % (REF_STEPS + 1) == REF_STEPS;
  const double tolS = last ? fmax(off_tol(L, l), 0x1p-53 * L.c[l]) : off_tol(L, l), tolP = 24.0 * 0x1p-53;
  const double pjj = re(p[j]), lj = pjj > 0.0 ? re(s[j]) / pjj : 0.0;
  double rho = 0.0;
  unsigned flag = 0;
  for (int i = lane; i < n; i += 32) {
    const T si = s[i], pi = p[i];
    if (i == j) {
      if (!(fabs(pjj - 1.0) <= tolP)) flag |= LEAF_OPEN | LEAF_SKEW;
      continue;
    }
    const double w = abs2(sub(si, scal(lj, pi)));
    if (!(w <= tolS * tolS)) flag |= LEAF_OPEN;
    if (!(abs2(pi) <= tolP * tolP)) flag |= LEAF_OPEN | LEAF_SKEW;
    rho += w;
  }
  rho = warp_sum(rho);
  flag = __reduce_or_sync(0xffffffffu, flag);
  if (lane == 0) {
    L.lam[L.voff[l] + j] = lj;
    L.rho[L.voff[l] + j] = sqrt(rho);
    if (flag) atomicOr(&L.off[l * OFF_N + it], flag);
  }
}

// The correction E.  A pair is rotated when its eigenvalues are further apart
// than GAP times the coupling of either column (then the rows of E have norm at
// most 1/4, X stays within some per cent of orthonormal and the step converges
// quadratically; with twice the coupling graded spectra lost orthonormality)
// and its coupling is above rounding; the others are only re-orthogonalised.
template <class T>
__global__ void leaf_correction_kernel(LeafDev L, int it, int ortho_only, const T* S, const T* P, T* E) {
  const int l = blockIdx.y, n = L.sz[l];
  if (leaf_ended(L, l, it)) return;
  const long long o = L.goff[l];
  const double *lam = L.lam + L.voff[l], *rho = L.rho + L.voff[l];
  const double tol = off_tol(L, l);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int i = e % n, j = e / n;
    const T p = P[o + e];
    T v;
    if (i == j) {
      v = from_re<T>(0.5 * (1.0 - re(p)));
    } else {
      // e_ij + conj(e_ji) = -p_ij: both entries of a pair take the same branch
      const T num = sub(S[o + e], scal(lam[j], p)), mirror = sub(S[o + e], scal(lam[i], p));
      const double den = lam[j] - lam[i];
      const bool apart = fabs(den) > GAP * fmax(rho[i], rho[j]);
      if (!ortho_only && apart && fmax(abs2(num), abs2(mirror)) > tol * tol) v = scal(1.0 / den, num);
      else v = scal(-0.5, p);
    }
    E[o + e] = v;
  }
}

// Next pass of stage 1, one CTA per open leaf: the columns in ascending order
// of lambda fall into clusters, cut where every column below is GAP couplings
// away from every column above, so that each pair which the refinement does not
// rotate is inside a cluster (a cut between neighbours that are far apart by
// their own couplings alone leaves pairs which nothing treats, and the passes
// stall); cluster k's shift (its mean lambda), scale (1 / Frobenius norm of
// its shifted block, from lambda and rho) and label.
__global__ void __launch_bounds__(1024) leaf_cluster_kernel(LeafDev L, int pass) {
  __shared__ double sl[LEAF_MAX], sr[LEAF_MAX], below[LEAF_MAX];
  __shared__ int start[LEAF_MAX];
  const int l = blockIdx.x, n = L.sz[l], tid = threadIdx.x;
  if (leaf_ended(L, l, pass * (REF_STEPS + 1) - 1)) return;
  const double *lam = L.lam + L.voff[l], *rho = L.rho + L.voff[l];
  int rank = 0;
  double li = 0.0, ri = 0.0;
  if (tid < n) {
    li = lam[tid];
    ri = rho[tid];
    for (int k = 0; k < n; ++k) rank += (lam[k] < li) || (lam[k] == li && k < tid) || (lam[k] != lam[k] && k < tid);
    rank = min(rank, n - 1);
    sl[rank] = li;
    sr[rank] = ri;
  }
  __syncthreads();
  if (tid == 0) {
    double lowest = INFINITY;  // of lambda - GAP rho over the columns from k on
    for (int k = n - 1; k >= 0; --k) below[k] = lowest = fmin(lowest, sl[k] - GAP * sr[k]);
    double highest = -INFINITY;  // of lambda + GAP rho over the columns before k
    int s0 = 0;
    for (int k = 0; k < n; ++k) {
      if (k > 0 && sl[k] > highest && below[k] > sl[k - 1]) s0 = k;
      highest = fmax(highest, sl[k] + GAP * sr[k]);
      start[k] = s0;
    }
  }
  __syncthreads();
  if (tid < n) {
    const int s0 = start[rank];
    double m = 0.0, f = 0.0;
    int e = s0;
    for (; e < n && start[e] == s0; ++e) m += sl[e];
    m /= e - s0;
    for (int k = s0; k < e; ++k) f += (sl[k] - m) * (sl[k] - m) + sr[k] * sr[k];
    L.label[L.voff[l] + tid] = s0;
    L.mean[L.voff[l] + tid] = m;
    L.scale[L.voff[l] + tid] = (e - s0 > 1 && f > 0.0) ? 1.0 / sqrt(f) : 0.0;
  }
}

// W_l = the cluster blocks of S, shifted and scaled, + 1.05 I (FP32)
template <class T>
__global__ void leaf_cluster_fill_kernel(LeafDev L, int pass, const T* S, int lds) {
  constexpr bool CX = sizeof(T) == 16;
  const int l = blockIdx.y, n = L.sz[l];
  if (leaf_ended(L, l, pass * (REF_STEPS + 1) - 1)) return;
  const J32Geom g = j32_geom(n, CX, lds);
  const long long o = L.goff[l], vo = L.voff[l];
  float* W = L.w32 + L.woff[l];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int i = e % n, j = e / n;
    T v = zero<T>();
    if (i == j) v = from_re<T>((re(S[o + e]) - L.mean[vo + j]) * L.scale[vo + j] + 1.05);
    else if (L.label[vo + i] == L.label[vo + j]) v = scal(L.scale[vo + j], S[o + e]);
    float* w = W + (long long)j * g.ldg + (CX ? 2 * i : i);
    w[0] = (float)re(v);
    if (CX) w[1] = (float)im(v);
  }
}

// X <- P for the leaves open at look `it`
template <class T>
__global__ void leaf_copy_kernel(LeafDev L, int it, const T* P, T* X) {
  const int l = blockIdx.y, n = L.sz[l];
  if (leaf_ended(L, l, it)) return;
  const long long o = L.goff[l];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) X[o + e] = P[o + e];
}

struct JRec {
  double c, s, phr, phi;
  int p, q, on, pad;
};

__device__ __forceinline__ double make_phase(double r, double, double) { return r; }
__device__ __forceinline__ z64 make_phase(double r, double i, z64) { return z64{r, i}; }

// Stage 3: two-sided cyclic Jacobi on G = S (tournament order), a cluster of
// JAC_CTAS CTAs per leaf; leaves that the refinement ended leave at once.  A
// round: the rotations of its disjoint pairs from the pivots of a CTA's own
// columns and their column rotations of G and V; cluster barrier; the row
// rotations of every pair on a CTA's own columns; cluster barrier.  Pairs
// with |g_pq| <= u ||B||_F are not rotated; a sweep with no rotation ends the
// leaf, which done[l] = 1 reports.
template <class T>
__global__ void __cluster_dims__(JAC_CTAS, 1, 1) __launch_bounds__(JAC_THREADS)
    leaf_jacobi_kernel(LeafDev L, const T* B, T* G_, T* V_, JRec* recs, int max_sweeps) {
  cg::cluster_group cluster = cg::this_cluster();
  const int l = blockIdx.x / JAC_CTAS, rank = blockIdx.x % JAC_CTAS, n = L.sz[l];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = JAC_THREADS / 32;
  if (n < 2 || leaf_ended(L, l, OFF_N - 1)) {  // uniform over the cluster
    if (rank == 0 && tid == 0) L.done[l] = 1;
    return;
  }
  T* G = G_ + L.goff[l];
  T* V = V_ + L.goff[l];
  JRec* rec = recs + L.roff[l];
  int* rot = L.rot + l * JAC_SWEEPS_MAX;
  const double thr = 0x1p-53 * L.c[l];
  const int np = n + (n & 1), pairs = np / 2;
  bool conv = false;
  if (L.off[l * OFF_N + OFF_N - 1] & LEAF_SKEW) {
    for (int e = rank * JAC_THREADS + tid; e < n * n; e += JAC_CTAS * JAC_THREADS) {
      G[e] = B[L.boff[l] + e % n + (long long)(e / n) * L.ldb[l]];
      V[e] = from_re<T>(e % n == e / n ? 1.0 : 0.0);
    }
    __threadfence();
    cluster.sync();
  }
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    for (int r = 0; r < np - 1; ++r) {
      for (int k = rank * nw + warp; k < pairs; k += JAC_CTAS * nw) {  // a warp per pair
        int p, q;
        tournament(np, r, k, p, q);
        JRec R{1.0, 0.0, 1.0, 0.0, p, q, 0, 0};
        if (q < n) {
          T* gp = G + (long long)p * n;
          T* gq = G + (long long)q * n;
          const double gpp = re(gp[p]), gqq = re(gq[q]);
          const T gpq = gq[p];
          __syncwarp();
          const double g = sqrt(abs2(gpq));
          if (g > thr) {
            const T ph = scal(1.0 / g, gpq);
            const double zeta = (gqq - gpp) / (2.0 * g);
            const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
            const double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
            R.c = c;
            R.s = s;
            R.phr = re(ph);
            R.phi = im(ph);
            R.on = 1;
            T* vp = V + (long long)p * n;
            T* vq = V + (long long)q * n;
            for (int i = lane; i < n; i += 32) {
              T x = gp[i], y = mul(gq[i], conj_(ph));
              gp[i] = sub(scal(c, x), scal(s, y));
              gq[i] = add(scal(s, x), scal(c, y));
              x = vp[i];
              y = mul(vq[i], conj_(ph));
              vp[i] = sub(scal(c, x), scal(s, y));
              vq[i] = add(scal(s, x), scal(c, y));
            }
            if (lane == 0) atomicAdd(&rot[sweep], 1);
          }
        }
        if (lane == 0) rec[k] = R;
      }
      __threadfence();
      cluster.sync();
      for (int k = tid; k < pairs; k += JAC_THREADS) {
        const JRec R = rec[k];
        if (!R.on) continue;
        const T ph = make_phase(R.phr, R.phi, T{});
        for (int j = rank; j < n; j += JAC_CTAS) {
          T* gc = G + (long long)j * n;
          const T x = gc[R.p], y = mul(gc[R.q], ph);
          gc[R.p] = sub(scal(R.c, x), scal(R.s, y));
          gc[R.q] = add(scal(R.s, x), scal(R.c, y));
        }
      }
      __threadfence();
      cluster.sync();
    }
    const int count = *(volatile int*)&rot[sweep];
    if (count == 0) {
      conv = true;
      break;
    }
  }
  if (rank == 0 && tid == 0) L.done[l] = conv ? 1 : 0;
}

// handle = 1 when a leaf is open at look `it` (one CTA)
__global__ void __launch_bounds__(256) leaf_any_open_kernel(LeafDev L, int it, cudaGraphConditionalHandle handle) {
  unsigned any = 0;
  for (int l = threadIdx.x; l < L.nl; l += blockDim.x) any |= L.off[l * OFF_N + it];
  any = __syncthreads_or(any != 0);
  if (threadIdx.x == 0) cudaGraphSetConditional(handle, any ? 1u : 0u);
}

// While cx.stream is captured: what body(s) launches on the stream s becomes
// the body of a conditional node, run when a leaf is open at look `it`.  A pass
// of 144 launches (256 rows) that nothing needs then costs one kernel; launched
// and left at once, as the second pass was, it took 0.2 ms.
template <class F>
void capture_if_open(Ctx& cx, const LeafDev& L, int it, F body) {
  cudaStreamCaptureStatus cs;
  cudaGraph_t graph = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  const cudaGraphEdgeData* edges = nullptr;
  size_t ndeps = 0;
  ZCSD_CUDA(cudaStreamGetCaptureInfo(cx.stream, &cs, nullptr, &graph, nullptr, nullptr, nullptr));
  cudaGraphConditionalHandle handle;
  ZCSD_CUDA(cudaGraphConditionalHandleCreate(&handle, graph, 0, cudaGraphCondAssignDefault));
  leaf_any_open_kernel<<<1, 256, 0, cx.stream>>>(L, it, handle);
  ZCSD_LAUNCH();
  ZCSD_CUDA(cudaStreamGetCaptureInfo(cx.stream, &cs, nullptr, &graph, &deps, &edges, &ndeps));
  cudaGraphNodeParams p = {};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = handle;
  p.conditional.type = cudaGraphCondTypeIf;
  p.conditional.size = 1;
  cudaGraphNode_t node;
  ZCSD_CUDA(cudaGraphAddNode(&node, graph, deps, edges, ndeps, &p));
  ZCSD_CUDA(cudaStreamUpdateCaptureDependencies(cx.stream, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
  cudaGraph_t inner = p.conditional.phGraph_out[0];
  ZCSD_CUDA(cudaStreamBeginCaptureToGraph(cx.body_stream, inner, nullptr, nullptr, 0,
                                          cudaStreamCaptureModeThreadLocal));
  body(cx.body_stream);
  ZCSD_CUDA(cudaStreamEndCapture(cx.body_stream, &inner));
}

// lambda[loff_l + j] = s_jj (blockIdx.y = leaf)
template <class T>
__global__ void leaf_values_kernel(LeafDev L, const T* G, double* lam) {
  const int l = blockIdx.y, n = L.sz[l];
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    lam[L.loff[l] + j] = re(G[L.goff[l] + j + (long long)j * n]);
}

template <bool CX, int NV>
void j32_launch(cudaStream_t st, const LeafTable& L, int pass, int sweep, int round, int ctas, bool chained) {
  constexpr int THREADS = j32_threads(128 * NV);
  static const bool attr = [] {
    ZCSD_CUDA(cudaFuncSetAttribute(j32_kernel<CX, NV, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, J32_SMEM));
    return true;
  }();
  (void)attr;
  const size_t smem = (size_t)L.maxcols * 128 * NV * 4;
  const dim3 grid(ctas, L.nl);
  if (chained)
    launch_chained(j32_kernel<CX, NV, THREADS>, grid, THREADS, smem, st, (const LeafDev&)L, pass, sweep, round);
  else j32_kernel<CX, NV, THREADS><<<grid, THREADS, smem, st>>>(L, pass, sweep, round);
  ZCSD_LAUNCH();
}

}  // namespace

LeafTable leaf_table_build(Ctx& cx, Arena& ar, const std::vector<long long>& boff, const std::vector<int>& ldb,
                           const std::vector<int>& loff, const std::vector<int>& sz, bool cplx) {
  LeafTable L;
  const int nl = (int)sz.size();
  L.nl = nl;
  for (int l = 0; l < nl; ++l) L.maxsz = std::max(L.maxsz, sz[l]);
  L.nv = std::max(1, ceil_div((cplx ? 2 : 1) * L.maxsz, 128));
  if (L.nv > 8) L.nv = L.nv <= 12 ? 12 : 16;  // complex leaves above 512 rows
  const int lds = 128 * L.nv;
  std::vector<int> hi(3 * nl, 0);
  std::vector<long long> hl(5 * nl + 4, 0);
  long long* hb = hl.data();
  long long *hg = hb + nl, *hw = hg + nl + 1, *hr = hw + nl + 1, *hv = hr + nl + 1;
  for (int l = 0; l < nl; ++l) {
    const J32Geom g = j32_geom(sz[l], cplx, lds);
    hi[l] = ldb[l];
    hi[nl + l] = loff[l];
    hi[2 * nl + l] = sz[l];
    hb[l] = boff[l];
    hg[l + 1] = hg[l] + (long long)sz[l] * sz[l];
    hw[l + 1] = hw[l] + (((long long)sz[l] * g.ldg + 63) & ~63LL);
    hr[l + 1] = hr[l] + (sz[l] + 1) / 2;
    hv[l + 1] = hv[l] + sz[l];
    L.maxblk = std::max(L.maxblk, g.nblk);
    L.maxcols = std::max(L.maxcols, 2 * g.wb);
  }
  L.vtot = hg[nl];
  L.hsz = sz;
  L.hldb = ldb;
  L.hboff = boff;
  L.hgoff.assign(hg, hg + nl);
  int* di = ar.get<int>(hi.size());
  long long* dl = ar.get<long long>(hl.size());
  ZCSD_CUDA(cudaMemcpyAsync(di, hi.data(), sizeof(int) * hi.size(), cudaMemcpyHostToDevice, cx.stream));
  ZCSD_CUDA(cudaMemcpyAsync(dl, hl.data(), sizeof(long long) * hl.size(), cudaMemcpyHostToDevice, cx.stream));
  ZCSD_CUDA(cudaStreamSynchronize(cx.stream));  // host tables go out of scope
  L.ldb = di;
  L.loff = di + nl;
  L.sz = di + 2 * nl;
  L.boff = dl;
  L.goff = dl + nl;
  L.woff = L.goff + nl + 1;
  L.roff = L.woff + nl + 1;
  L.voff = L.roff + nl + 1;
  L.c = ar.get<double>(nl);
  L.done = ar.get<int>(nl);
  L.rot = ar.get<int>((size_t)nl * JAC_SWEEPS_MAX);
  L.cosmax = ar.get<int>((size_t)nl * PASSES * J32_SWEEPS);
  L.off = ar.get<unsigned>((size_t)nl * OFF_N);
  L.lam = ar.get<double>(4 * (size_t)hv[nl]);
  L.rho = L.lam + hv[nl];
  L.mean = L.rho + hv[nl];
  L.scale = L.mean + hv[nl];
  L.label = ar.get<int>((size_t)hv[nl]);
  L.x32 = ar.get<float>(4 * (size_t)hv[nl]);
  L.part = ar.get<double>((size_t)nl * 2 * PRE_PARTS);
  L.norms = ar.get<double>((size_t)nl * 2);
  L.w32 = ar.get<float>((size_t)hw[nl]);
  L.recs = ar.get<char>((size_t)hr[nl] * sizeof(JRec));
  return L;
}

size_t leaf_table_bytes(const std::vector<int>& sz, bool cplx) {
  size_t b = 24 * 256, f = cplx ? 2 : 1;
  for (int s : sz)
    b += (size_t)s * (f * s + 4) * 4 + 256 + (size_t)(s + 1) / 2 * sizeof(JRec) + 3 * 4 + 4 * 8 + 12 +
         JAC_SWEEPS_MAX * 4 + PASSES * J32_SWEEPS * 4 + OFF_N * 4 + 52 * (size_t)s + 8 + 16 * PRE_PARTS + 16;
  return b;
}

template <class T>
void leaf_solve(Ctx& cx, Arena& ar, const LeafTable& L, const T* B, double* lam, T* V, int max_sweeps,
                bool sync_free) {
  constexpr bool CX = sizeof(T) == 16;
  cudaStream_t st = cx.stream;
  if (L.nl == 0) return;
  const size_t mk = ar.mark();
  T* Tm = ar.get<T>((size_t)L.vtot);
  T* S = ar.get<T>((size_t)L.vtot);
  T* P = ar.get<T>((size_t)L.vtot);
  ProfToken tok = prof_begin(st);
  const int lds = 128 * L.nv;
  leaf_norm_kernel<T><<<dim3(PRE_PARTS, L.nl), 256, 0, st>>>(L, B);
  ZCSD_LAUNCH();
  leaf_fill_kernel<T><<<dim3(std::max(1, std::min(ceil_div((long long)L.maxsz * L.maxsz, 1024), 152)), L.nl), 256, 0,
                        st>>>(L, B, lds);
  ZCSD_LAUNCH();
  for (int it = 0; it <= POW_STEPS; ++it) {
    leaf_power_kernel<CX><<<dim3(ceil_div(L.maxsz, 8), L.nl), 256, 0, st>>>(L, it, lds);
    ZCSD_LAUNCH();
  }
  const int tiles = ceil_div(L.maxsz, MM_R) * ceil_div(L.maxsz, MM_C);
  const int ew = std::max(1, std::min(ceil_div((long long)L.maxsz * L.maxsz, 256), 304));
  const dim3 cols(ceil_div(L.maxsz, 8), L.nl);
  // Leaves of LEAF_TC rows and more take their products from gemm() when the
  // tensor cores are on (there a product costs launches and conversions, here
  // n^3 on the FP64 pipe).  A call that may be captured keeps to one launch for
  // all leaves.
  std::vector<int> big;
  if (!sync_free && t_tc.enabled)
    for (int l = 0; l < L.nl; ++l)
      if (L.hsz[l] >= LEAF_TC) big.push_back(l);
  const int max_n = big.empty() ? LEAF_MAX : LEAF_TC - 1;
  const T one = from_re<T>(1.0), zer = zero<T>();
  std::vector<unsigned> hoff((size_t)L.nl * OFF_N, 1u);
  auto open = [&](int l, int look) { return look < 0 || hoff[(size_t)l * OFF_N + look] != 0u; };
  auto read_state = [&](int look) {
    ZCSD_CUDA(cudaMemcpyAsync(hoff.data(), L.off, sizeof(unsigned) * hoff.size(), cudaMemcpyDeviceToHost, st));
    ZCSD_CUDA(cudaStreamSynchronize(st));
    bool any = false;
    for (int l = 0; l < L.nl; ++l) any = any || open(l, look);
    return any;
  };
  auto mul_big = [&](int look, int opA, const T* A, const T* Bm, T* C, bool fromB, T beta) {
    for (int l : big) {
      if (!open(l, look)) continue;
      const int n = L.hsz[l];
      const long long o = L.hgoff[l];
      if (fromB) gemm1<T>(st, opA, OP_N, n, n, n, one, A + L.hboff[l], L.hldb[l], Bm + o, n, beta, C + o, n, 0, 0, GS_EIG);
      else gemm1<T>(st, opA, OP_N, n, n, n, one, A + o, n, Bm + o, n, beta, C + o, n, 0, 0, GS_EIG);
    }
  };
  // one pass on the stream s; false once every leaf has ended, where the host
  // may read that
  auto run_pass = [&](int pass, cudaStream_t s, bool reads) -> bool {
    bool any = true;
    // two steps more of the kind at the end: stage 3 starts from S only where X is orthonormal
    const int ortho = pass + 1 < PASSES ? ORTHO_STEPS : 2 * ORTHO_STEPS;
    const int look0 = pass * (REF_STEPS + 1);
    if (pass > 0) {
      leaf_cluster_kernel<<<L.nl, 1024, 0, s>>>(L, pass);
      ZCSD_LAUNCH();
      leaf_cluster_fill_kernel<T><<<dim3(ew, L.nl), 256, 0, s>>>(L, pass, S, lds);
      ZCSD_LAUNCH();
    }
    const bool one_cta = L.maxblk == 2;
    for (int sweep = 0; sweep < (one_cta ? 1 : J32_SWEEPS); ++sweep) {
      for (int r = 0; r < L.maxblk - 1; ++r) {
        switch (L.nv) {
#define ZCSD_J32(NV) case NV: j32_launch<CX, NV>(s, L, pass, sweep, r, L.maxblk / 2, s == st); break;
          ZCSD_J32(1) ZCSD_J32(2) ZCSD_J32(3) ZCSD_J32(4) ZCSD_J32(5) ZCSD_J32(6) ZCSD_J32(7) ZCSD_J32(8)
          default:
            if constexpr (CX) {
              if (L.nv == 12) j32_launch<CX, 12>(s, L, pass, sweep, r, L.maxblk / 2, s == st);
              else j32_launch<CX, 16>(s, L, pass, sweep, r, L.maxblk / 2, s == st);
            }
#undef ZCSD_J32
        }
      }
    }
    leaf_basis_kernel<T><<<cols, 256, 0, s>>>(L, pass, pass == 0 ? V : Tm, lds);
    ZCSD_LAUNCH();
    if (pass > 0) {  // X <- X Y
      leaf_mm_kernel<T, MM_XY><<<dim3(tiles, L.nl), MM_R * MM_C, 0, s>>>(L, look0, max_n, B, V, Tm, S, P);
      ZCSD_LAUNCH();
      mul_big(look0 - 1, OP_N, V, Tm, P, false, zer);
      leaf_copy_kernel<T><<<dim3(ew, L.nl), 256, 0, s>>>(L, look0 - 1, P, V);
      ZCSD_LAUNCH();
    }
    for (int it = 0; it <= REF_STEPS; ++it) {
      const int look = look0 + it;
      leaf_mm_kernel<T, MM_BX><<<dim3(tiles, L.nl), MM_R * MM_C, 0, s>>>(L, look, max_n, B, V, Tm, S, P);
      ZCSD_LAUNCH();
      mul_big(look - 1, OP_N, B, V, Tm, true, zer);
      leaf_mm_kernel<T, MM_GRAM><<<dim3(tiles, L.nl, 2), MM_R * MM_C, 0, s>>>(L, look, max_n, B, V, Tm, S, P);
      ZCSD_LAUNCH();
      mul_big(look - 1, OP_C, V, Tm, S, false, zer);
      mul_big(look - 1, OP_C, V, V, P, false, zer);
      leaf_state_kernel<T><<<cols, 256, 0, s>>>(L, look, S, P);
      ZCSD_LAUNCH();
      // stop once every leaf has ended (rarely before the third look)
      if (reads && (it >= 2 || !big.empty()) && !(any = read_state(look))) break;
      if (it == REF_STEPS) break;
      leaf_correction_kernel<T><<<dim3(ew, L.nl), 256, 0, s>>>(L, look, it >= REF_STEPS - ortho, S, P, Tm);
      ZCSD_LAUNCH();
      leaf_mm_kernel<T, MM_XE><<<dim3(tiles, L.nl), MM_R * MM_C, 0, s>>>(L, look, max_n, B, V, Tm, S, P);
      ZCSD_LAUNCH();
      if (!big.empty()) {
        for (int l : big)
          if (open(l, look))
            axpby<T>(st, L.hsz[l], L.hsz[l], 1.0, V + L.hgoff[l], L.hsz[l], 0, 0.0, P + L.hgoff[l], L.hsz[l], 0, 1);
        mul_big(look, OP_N, V, Tm, P, false, one);
      }
      leaf_copy_kernel<T><<<dim3(ew, L.nl), 256, 0, s>>>(L, look, P, V);
      ZCSD_LAUNCH();
    }
    return any;
  };
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (sync_free) ZCSD_CUDA(cudaStreamIsCapturing(st, &cs));
  if (cs == cudaStreamCaptureStatusNone) {
    for (int pass = 0; pass < PASSES && run_pass(pass, st, true); ++pass) {
    }
  } else {
    run_pass(0, st, false);
    for (int pass = 1; pass < PASSES; ++pass)
      capture_if_open(cx, L, pass * (REF_STEPS + 1) - 1, [&](cudaStream_t s) { run_pass(pass, s, false); });
  }
  leaf_jacobi_kernel<T><<<L.nl * JAC_CTAS, JAC_THREADS, 0, st>>>(L, B, S, V, reinterpret_cast<JRec*>(L.recs),
                                                                 std::min(max_sweeps, (int)JAC_SWEEPS_MAX));
  ZCSD_LAUNCH();
  leaf_values_kernel<T><<<dim3(ceil_div(L.maxsz, 256), L.nl), 256, 0, st>>>(L, S, lam);
  ZCSD_LAUNCH();
  if (tok.slot >= 0) prof_end(tok, st, PK_JACOBI, 0.0);
  ar.release(mk);
}

template void leaf_solve<double>(Ctx&, Arena&, const LeafTable&, const double*, double*, double*, int, bool);
template void leaf_solve<z64>(Ctx&, Arena&, const LeafTable&, const z64*, double*, z64*, int, bool);

template <class T>
void jacobi_eig_leaves(Ctx& cx, Arena& ar, const std::vector<int>& off, const std::vector<int>& sz, const T* B,
                       int ldb, double* lam, T* Vl, std::vector<long long>& voff) {
  const int nl = (int)off.size();
  if (nl == 0) return;
  const size_t mk = ar.mark();
  std::vector<long long> boff(nl);
  std::vector<int> lds(nl, ldb);
  voff.assign(nl + 1, 0);
  for (int l = 0; l < nl; ++l) {
    boff[l] = off[l] + (long long)off[l] * ldb;
    voff[l + 1] = voff[l] + (long long)sz[l] * sz[l];
  }
  const LeafTable L = leaf_table_build(cx, ar, boff, lds, off, sz, sizeof(T) == 16);
  leaf_solve<T>(cx, ar, L, B, lam, Vl, JAC_SWEEPS_MAX, false);
  ar.release(mk);
}

template void jacobi_eig_leaves<double>(Ctx&, Arena&, const std::vector<int>&, const std::vector<int>&, const double*,
                                        int, double*, double*, std::vector<long long>&);
template void jacobi_eig_leaves<z64>(Ctx&, Arena&, const std::vector<int>&, const std::vector<int>&, const z64*, int,
                                     double*, z64*, std::vector<long long>&);

}  // namespace zcsd
