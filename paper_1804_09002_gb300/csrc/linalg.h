// Blocked factorizations built from the kernels of blas.cu / fact.cu, and the
// device workspace arena they draw from.  Host-side orchestration only.
#pragma once
#include <algorithm>
#include <vector>

#include "ops.h"

namespace zcsd {

constexpr int NB_QR = 32;    // Householder panel width
constexpr int NB_OUT = 128;  // outer block of the two-level blocked QR
constexpr int LEAF = 1024;   // Zolo-eig leaf size, default (leaf.cu: a 1024-row leaf is faster than one split of it)
constexpr int LEAF_MAX = 1024;  // largest leaf size a context may set

struct ArenaOverflow {
  size_t needed;
};

// Bump allocator over one device allocation, with stack-like mark/release.
struct Arena {
  char* base = nullptr;
  size_t cap = 0, off = 0, peak = 0;
  template <class X>
  X* get(size_t count) {
    size_t bytes = (count * sizeof(X) + 255) & ~(size_t)255;
    if (off + bytes > cap) throw ArenaOverflow{off + bytes};
    X* p = reinterpret_cast<X*>(base + off);
    off += bytes;
    peak = std::max(peak, off);
    return p;
  }
  size_t mark() const { return off; }
  void release(size_t m) { off = m; }
};

// Pinned host scratch for device->host scalars.
struct HostScalars {
  double* d = nullptr;  // pinned, 64 doubles
  int* i = nullptr;     // pinned, 4096 ints
};

// ---- Householder QR of `batch` m x n matrices M_b (ld ldm, stride sM) in
// which the reflector of column k spans rows [k, min(m, k + band)).  On
// return M holds R (upper) and the reflectors (below); QRStore keeps the
// explicit V panels and T factors for applying / forming Q.
template <class T>
struct QRStore {
  int m = 0, n = 0, band = 0, batch = 0, npan = 0, ldy = 0, nbo = 0;
  T* Y = nullptr;  // per problem: npan outer blocks of ldy x nbo (nbo = min(NB_OUT, n rounded up to 32))
  T* Tf = nullptr; // per problem: npan blocks of nbo x nbo
  long long sY = 0, sT = 0;
};

template <class T> QRStore<T> qr_alloc(Arena& ar, int m, int n, int band, int batch);
template <class T> void qr_factor(cudaStream_t st, Arena& ar, QRStore<T>& q, T* M, int ldm, long long sM);
// E_b = Q_b [I; 0] (m x n, ld lde, stride sE)
template <class T> void qr_form_q(cudaStream_t st, Arena& ar, const QRStore<T>& q, T* E, int lde, long long sE);

// ---- N_b = R_b^{-1}, the inverse of the upper Cholesky factor R^* R = Z_b, of
// `batch` n x n matrices.  Z's upper triangle is overwritten; N must be zero
// below its diagonal on entry (it stays so).
template <class T>
void chol_inverse(cudaStream_t st, Arena& ar, int n, T* Z, int ldz, long long sZ, T* N, int ldn, long long sN,
                  int batch);

// ---- C = alpha sum_j w_j op(A_j) op(B_j) + beta Cin, as gemm(); complex sums
// go term by term where that lets the tensor cores take them.
template <class T>
void gemm_terms(GemmArgs<T> g, cudaStream_t st);

}  // namespace zcsd
