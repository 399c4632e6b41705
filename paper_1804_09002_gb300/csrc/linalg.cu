// Blocked Householder QR (compact WY) and the recursive inverse Cholesky
// factor, as sequences of panel kernels and batched GEMMs.
#include <type_traits>

#include "linalg.h"
#include "tc_gemm.h"

namespace zcsd {

// Split-K factor for a product whose output alone gives too few tiles, or a
// tile count that fills its last wave poorly, for tiles of 4096 outputs (gemm()
// may take smaller ones, which need less of a split): the GEMM keeps two CTAs per SM
// resident (304 slots on 152 SMs), so a launch of C CTAs runs ceil(C / 304)
// waves; pick the split s (K chunks of at least kmin) that maximises the
// filled fraction C s / (304 ceil(C s / 304)), smaller s on ties.
static int pick_ksplit(int m, int n, int k, int batch, int bm, int kmin = 256) {
  const long long tiles = (long long)ceil_div(m, bm) * ceil_div(n, 4096 / bm) * batch;
  const int smax = std::min(MAX_SUM, std::max(1, k / kmin));
  constexpr long long slots = 2 * 152;
  int best = 1;
  double best_eff = -1.0;
  for (int s = 1; s <= smax; ++s) {
    const long long c = tiles * s;
    const double eff = (double)c / (double)(slots * ((c + slots - 1) / slots));
    if (eff > best_eff + 0.02) {
      best_eff = eff;
      best = s;
    }
  }
  return best;
}

// Split-K factor of a product: the FP64-pipe choice `ks`, at most `cap`, the
// partial buffers the caller holds, or 1 when the tensor-core path takes the
// product (its items, one per modulus, fill the SMs).
template <class T>
static int resolve_ksplit(GemmArgs<T>& g, int ks, int cap) {
  g.ksplit = std::max(1, std::min(ks, cap));
  GemmArgs<T> probe = g;
  probe.ksplit = 1;
  if constexpr (std::is_same<T, double>::value) {
    if (tc_will_handle(probe)) g.ksplit = 1;
  } else {
    if (tc_will_handle_complex(probe)) g.ksplit = 1;
  }
  return g.ksplit;
}

template <class T>
QRStore<T> qr_alloc(Arena& ar, int m, int n, int band, int batch) {
  QRStore<T> q;
  q.m = m; q.n = n; q.band = band; q.batch = batch;
  q.nbo = std::min(NB_OUT, ceil_div(n, NB_QR) * NB_QR);  // outer block width (small n: the whole matrix)
  q.npan = ceil_div(n, q.nbo);
  q.ldy = std::max(1, std::min(m, q.nbo - 1 + band));
  q.sY = (long long)q.npan * q.ldy * q.nbo;
  q.sT = (long long)q.npan * q.nbo * q.nbo;
  q.Y = ar.get<T>((size_t)q.sY * batch);
  q.Tf = ar.get<T>((size_t)q.sT * batch);
  return q;
}

// C <- (I - Y op(T) Y^*) C for `batch` problems: op(T) = T^* applies Q^* (the
// factorization sweep), op(T) = T applies Q (forming Q).  Y is h x nb with
// explicit zeros / unit diagonal, T is nb x nb upper triangular, C is h x nc.
// W = Y^* C is split along its long K = h range when its output is small.
template <class T>
static void wy_apply(cudaStream_t st, Arena& ar, int h, int nc, int nb, const T* Y, int ldy, long long sY,
                     const T* Tm, int ldt, long long sT, bool adjoint, T* C, int ldc, long long sC, int batch,
                     int site_w, int site_w2, int site_upd) {
  if (nc <= 0 || nb <= 0 || h <= 0) return;
  const int kcap = std::min(nb > NB_QR ? 4 : MAX_SUM, std::max(1, h / 256));
  const size_t mk = ar.mark();
  const long long sW = (long long)nb * nc;
  T* W = ar.get<T>((size_t)sW * batch * kcap);
  T* W2 = ar.get<T>((size_t)sW * batch);
  const T one = from_re<T>(1.0), mone = from_re<T>(-1.0), zer = zero<T>();
  GemmArgs<T> g;  // W_s = Y^* C over K chunk s
  g.batch = batch;
  g.m = nb; g.n = nc; g.k = h; g.opA = OP_C; g.opB = OP_N;
  g.A = Y; g.lda = ldy; g.sA = sY;
  g.B = C; g.ldb = ldc; g.sB = sC;
  g.C = W; g.ldc = nb; g.sC = sW;
  g.site = site_w;
  g.alpha = one; g.beta = zer;
  const int ks = resolve_ksplit(g, pick_ksplit(nb, nc, h, batch, nb <= 32 ? 32 : 64), kcap);
  gemm(g, st);
  sum_parts<T>(st, nb, nc, W, nb, sW, ks, batch);  // W_0 = sum_s W_s
  GemmArgs<T> g2;  // W2 = op(T) W_0
  g2.batch = batch;
  g2.m = nb; g2.n = nc; g2.k = nb;
  g2.opA = adjoint ? OP_C : OP_N;
  g2.kflags = adjoint ? K_TO_ROW : K_FROM_ROW;  // T upper triangular
  g2.A = Tm; g2.lda = ldt; g2.sA = sT;
  g2.B = W; g2.ldb = nb; g2.sB = sW * ks;
  g2.C = W2; g2.ldc = nb; g2.sC = sW;
  g2.site = site_w2;
  g2.alpha = one; g2.beta = zer;
  gemm(g2, st);
  // C -= Y W2
  GemmArgs<T> g3;
  g3.batch = batch;
  g3.m = h; g3.n = nc; g3.k = nb; g3.opA = OP_N; g3.opB = OP_N;
  g3.A = Y; g3.lda = ldy; g3.sA = sY;
  g3.B = W2; g3.ldb = nb; g3.sB = sW;
  g3.Cin = C; g3.ldcin = ldc; g3.sCin = sC;
  g3.C = C; g3.ldc = ldc; g3.sC = sC;
  g3.site = site_upd;
  g3.kbal = 1;  // rows of any size: balance k on the tensor cores
  g3.alpha = mone; g3.beta = one;
  gemm(g3, st);
  ar.release(mk);
}

// Two-level blocked Householder QR: outer blocks of NB_OUT columns, each
// factored as NB_QR-wide panels (panel kernel + updates inside the block);
// the block's compact-WY factor T (NB_OUT x NB_OUT) is merged from the panel
// factors, T_{<i, i} = -T_{<i} (Y_{<i}^* Y_i) T_i (Q = Q_{<i} Q_i), and the
// trailing matrix is updated once per outer block.
template <class T>
void qr_factor(cudaStream_t st, Arena& ar, QRStore<T>& q, T* M, int ldm, long long sM) {
  const int m = q.m, n = q.n;
  const size_t mk = ar.mark();
  T* Tin = ar.get<T>((size_t)NB_QR * NB_QR * q.batch);
  const int NBO = q.nbo;
  const int scap = std::min(MAX_SUM, std::max(1, q.ldy / 256));
  T* S = ar.get<T>((size_t)NBO * NBO * q.batch * scap);  // split-K parts of the Gram matrix Y_b^* Y_b
  T* S2 = ar.get<T>((size_t)NBO * NB_QR * q.batch);
  const long long sS = (long long)NBO * NBO, sS2 = (long long)NBO * NB_QR;
  const T one = from_re<T>(1.0), mone = from_re<T>(-1.0), zer = zero<T>();
  for (int ob = 0; ob < q.npan; ++ob) {
    const int K0 = ob * NBO;
    if (K0 >= m) break;
    const int nbo = std::min(NBO, n - K0);
    const int hb = std::min(m, K0 + nbo - 1 + q.band) - K0;
    T* Yb = q.Y + (long long)ob * q.ldy * NBO;
    T* Tb = q.Tf + (long long)ob * NBO * NBO;
    ZCSD_CUDA(cudaMemset2DAsync(Yb, sizeof(T) * q.sY, 0, sizeof(T) * (size_t)q.ldy * NBO, q.batch, st));
    ZCSD_CUDA(cudaMemset2DAsync(Tb, sizeof(T) * q.sT, 0, sizeof(T) * (size_t)NBO * NBO, q.batch, st));
    for (int c0 = 0; c0 < nbo; c0 += NB_QR) {
      const int k0 = K0 + c0;
      if (k0 >= m) break;
      const int nb = std::min(NB_QR, nbo - c0);
      T* Yi = Yb + c0 + (long long)c0 * q.ldy;
      T* Ti = Tb + c0 + (long long)c0 * NBO;
      qr_panel<T>(st, m, n, q.band, M, ldm, sM, k0, nb, Yi, q.ldy, q.sY, Tin, (long long)NB_QR * NB_QR, q.batch);
      axpby<T>(st, nb, nb, 1.0, Tin, nb, (long long)NB_QR * NB_QR, 0.0, Ti, NBO, q.sT, q.batch);
      // update the rest of this outer block with panel i
      const int nc_in = K0 + nbo - (k0 + nb);
      if (nc_in > 0) {
        const int hi = std::min(m, k0 + nb - 1 + q.band) - k0;
        wy_apply<T>(st, ar, hi, nc_in, nb, Yi, q.ldy, q.sY, Ti, NBO, q.sT, true, M + k0 + (long long)(k0 + nb) * ldm,
                    ldm, sM, q.batch, GS_QR_W, GS_QR_W2, GS_QR_UPD);
      }
    }
    // merge the panel factors into the block's T: one Gram matrix
    // S = Y_b^* Y_b (split along its long K), then for each panel i,
    // T_{<i, i} = -T_{<i} S[<i, i] T_i  (Q = Q_{<i} Q_i)
    if (nbo > NB_QR) {
      GemmArgs<T> g;
      g.batch = q.batch;
      g.m = nbo; g.n = nbo; g.k = hb; g.opA = OP_C; g.opB = OP_N;
      g.A = Yb; g.lda = q.ldy; g.sA = q.sY;
      g.B = Yb; g.ldb = q.ldy; g.sB = q.sY;
      g.C = S; g.ldc = NBO; g.sC = sS;
      g.alpha = one; g.beta = zer; g.site = GS_TMERGE;
      const int ks = resolve_ksplit(g, pick_ksplit(nbo, nbo, hb, q.batch, 64), scap);
      gemm(g, st);
      sum_parts<T>(st, nbo, nbo, S, NBO, sS, ks, q.batch);  // S_0 = sum_s S_s
      for (int c0 = NB_QR; c0 < nbo; c0 += NB_QR) {
        const int nb = std::min(NB_QR, nbo - c0);
        T* Ti = Tb + c0 + (long long)c0 * NBO;
        GemmArgs<T> g2;  // S2 = T_{<i} S_0[<i, i]
        g2.batch = q.batch;
        g2.m = c0; g2.n = nb; g2.k = c0; g2.opA = OP_N; g2.opB = OP_N;
        g2.A = Tb; g2.lda = NBO; g2.sA = q.sT;
        g2.B = S + (long long)c0 * NBO; g2.ldb = NBO; g2.sB = sS * ks;
        g2.C = S2; g2.ldc = NBO; g2.sC = sS2;
        g2.alpha = one; g2.beta = zer; g2.kflags = K_FROM_ROW; g2.site = GS_TMERGE;
        gemm(g2, st);
        GemmArgs<T> g3;  // T_{<i, i} = -S2 T_i
        g3.batch = q.batch;
        g3.m = c0; g3.n = nb; g3.k = nb; g3.opA = OP_N; g3.opB = OP_N;
        g3.A = S2; g3.lda = NBO; g3.sA = sS2;
        g3.B = Ti; g3.ldb = NBO; g3.sB = q.sT;
        g3.C = Tb + (long long)c0 * NBO; g3.ldc = NBO; g3.sC = q.sT;
        g3.alpha = mone; g3.beta = zer; g3.kflags = K_TO_COL; g3.site = GS_TMERGE;
        gemm(g3, st);
      }
    }
    const int nc = n - (K0 + nbo);
    if (nc > 0)
      wy_apply<T>(st, ar, hb, nc, nbo, Yb, q.ldy, q.sY, Tb, NBO, q.sT, true, M + K0 + (long long)(K0 + nbo) * ldm,
                  ldm, sM, q.batch, GS_QR_W, GS_QR_W2, GS_QR_UPD);
  }
  ar.release(mk);
}

template <class T>
void qr_form_q(cudaStream_t st, Arena& ar, const QRStore<T>& q, T* E, int lde, long long sE) {
  const int m = q.m, n = q.n;
  set_eye<T>(st, m, n, E, lde, sE, q.batch);
  const int NBO = q.nbo;
  for (int ob = q.npan - 1; ob >= 0; --ob) {
    const int K0 = ob * NBO;
    if (K0 >= m) continue;
    const int nbo = std::min(NBO, n - K0);
    const int hb = std::min(m, K0 + nbo - 1 + q.band) - K0;
    const T* Yb = q.Y + (long long)ob * q.ldy * NBO;
    const T* Tb = q.Tf + (long long)ob * NBO * NBO;
    wy_apply<T>(st, ar, hb, n - K0, nbo, Yb, q.ldy, q.sY, Tb, NBO, q.sT, false, E + K0 + (long long)K0 * lde, lde,
                sE, q.batch, GS_FQ_W, GS_FQ_W2, GS_FQ_UPD);
  }
}

// Columns [c0, c1) of N = R^{-1}, R^* R = Z: invert the leading half, W =
// N11^* Z12 (= R12), Z22 -= W^* W, invert the trailing half, N12 = -N11 W N22.
// The factor itself is never formed, and no triangular system is solved:
// every step above the innermost blocks is a product with K = half the width.
template <class T>
static void chol_inv_rec(cudaStream_t st, Arena& ar, int c0, int c1, T* Z, int ldz, long long sZ, T* N, int ldn,
                         long long sN, int batch) {
  const int w = c1 - c0;
  if (w <= CHOL_NB) {
    chol_inv_block<T>(st, w, Z + c0 + (long long)c0 * ldz, ldz, sZ, N + c0 + (long long)c0 * ldn, ldn, sN, batch);
    return;
  }
  const int mid = c0 + ceil_div(w / 2, CHOL_NB) * CHOL_NB, w1 = mid - c0, w2 = c1 - mid;
  const T one = from_re<T>(1.0), mone = from_re<T>(-1.0), zer = zero<T>();
  chol_inv_rec(st, ar, c0, mid, Z, ldz, sZ, N, ldn, sN, batch);
  const size_t mk = ar.mark();
  const long long sW = (long long)w1 * w2;
  T* W = ar.get<T>((size_t)sW * batch);
  T* N11 = N + c0 + (long long)c0 * ldn;
  GemmArgs<T> g;  // W = N11^* Z12
  g.batch = batch;
  g.m = w1; g.n = w2; g.k = w1; g.opA = OP_C; g.opB = OP_N; g.kflags = K_TO_ROW;
  g.A = N11; g.lda = ldn; g.sA = sN;
  g.B = Z + c0 + (long long)mid * ldz; g.ldb = ldz; g.sB = sZ;
  g.C = W; g.ldc = w1; g.sC = sW;
  g.alpha = one; g.beta = zer; g.site = GS_CHOL_INV;
  gemm(g, st);
  GemmArgs<T> h;  // Z22 -= W^* W (tiles touching the upper triangle)
  h.batch = batch;
  h.m = w2; h.n = w2; h.k = w1; h.opA = OP_C; h.opB = OP_N; h.uplo = 1;
  h.A = W; h.lda = w1; h.sA = sW;
  h.B = W; h.ldb = w1; h.sB = sW;
  T* Z22 = Z + mid + (long long)mid * ldz;
  h.Cin = Z22; h.ldcin = ldz; h.sCin = sZ;
  h.C = Z22; h.ldc = ldz; h.sC = sZ;
  h.alpha = mone; h.beta = one; h.site = GS_CHOL_TRAIL;
  gemm(h, st);
  chol_inv_rec(st, ar, mid, c1, Z, ldz, sZ, N, ldn, sN, batch);
  T* V = ar.get<T>((size_t)sW * batch);
  GemmArgs<T> v;  // V = W N22
  v.batch = batch;
  v.m = w1; v.n = w2; v.k = w2; v.opA = OP_N; v.opB = OP_N; v.kflags = K_TO_COL;
  v.A = W; v.lda = w1; v.sA = sW;
  v.B = N + mid + (long long)mid * ldn; v.ldb = ldn; v.sB = sN;
  v.C = V; v.ldc = w1; v.sC = sW;
  v.alpha = one; v.beta = zer; v.site = GS_CHOL_INV;
  gemm(v, st);
  GemmArgs<T> u;  // N12 = -N11 V
  u.batch = batch;
  u.m = w1; u.n = w2; u.k = w1; u.opA = OP_N; u.opB = OP_N; u.kflags = K_FROM_ROW;
  u.A = N11; u.lda = ldn; u.sA = sN;
  u.B = V; u.ldb = w1; u.sB = sW;
  u.C = N + c0 + (long long)mid * ldn; u.ldc = ldn; u.sC = sN;
  u.alpha = mone; u.beta = zer; u.site = GS_CHOL_INV;
  gemm(u, st);
  ar.release(mk);
}

template <class T>
void chol_inverse(cudaStream_t st, Arena& ar, int n, T* Z, int ldz, long long sZ, T* N, int ldn, long long sN,
                  int batch) {
  chol_inv_rec<T>(st, ar, 0, n, Z, ldz, sZ, N, ldn, sN, batch);
}

template <class T>
void gemm_terms(GemmArgs<T> g, cudaStream_t st) {
  if constexpr (std::is_same<T, z64>::value) {
    GemmArgs<T> one = g;
    one.nsum = 1;
    if (g.nsum > 1 && tc_will_handle_complex(one)) {
      for (int j = 0; j < g.nsum; ++j) {
        one.A = g.A + j * g.sAj;
        one.B = g.B + j * g.sBj;
        one.alpha = scal(g.w[j], g.alpha);
        if (j > 0) {
          one.Cin = g.C; one.ldcin = g.ldc; one.sCin = g.sC;
          one.beta = from_re<T>(1.0);
        }
        gemm(one, st);
      }
      return;
    }
  }
  gemm(g, st);
}

#define ZCSD_INST_L(T)                                                                                          \
  template QRStore<T> qr_alloc<T>(Arena&, int, int, int, int);                                                  \
  template void qr_factor<T>(cudaStream_t, Arena&, QRStore<T>&, T*, int, long long);                            \
  template void qr_form_q<T>(cudaStream_t, Arena&, const QRStore<T>&, T*, int, long long);                      \
  template void chol_inverse<T>(cudaStream_t, Arena&, int, T*, int, long long, T*, int, long long, int);         \
  template void gemm_terms<T>(GemmArgs<T>, cudaStream_t);

ZCSD_INST_L(double)
ZCSD_INST_L(z64)

}  // namespace zcsd
