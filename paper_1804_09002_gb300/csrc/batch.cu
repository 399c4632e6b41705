// Many real FP64 CS decompositions of different sizes in one graph-captured
// launch (csd_batch_*).  The paper's only parallelism is between the two
// polar decompositions and the r terms of Zolo-pd (Section 3, remark (ii));
// here independent CSDs are batched as well:
//
//  * instances are grouped into buckets of padded size nb (a multiple of the
//    bucket granularity); inside a bucket every polar problem is the n x n
//    block embedded as diag(A_i, I): Zolo-pd's QR and Cholesky forms keep
//    that block structure exactly, so the padded problems return
//    diag(W_i, I) and one zolo_pd call serves both blocks of every CSD of
//    the bucket (the sync-free form: no host read between its launches);
//  * H_i = sym(W_i^* A_i) and B = H_2 - H_1 per instance (the padded part of
//    B is exactly zero), and every B of every bucket is one leaf of the
//    batched leaf eigensolver (leaf.cu) at its own size, with device-side
//    convergence flags;
//  * C, S = diag(V^* H_i V), theta = atan2(S, C), U_i = W_i V by batched
//    products on the padded V, then one CTA per instance sorts its angles
//    and writes its columns into the packed outputs.
//
// Everything between the input and the output buffers runs with no host
// synchronisation, so the whole batch is captured once into a CUDA graph and
// replayed.  A bucket is a chain of small launches that leaves most SMs idle,
// and buckets share nothing but read-only inputs, so they run side by side on
// up to MAX_LANES streams, each with its own part of the workspace (48
// instances of 16..256 rows in 16 buckets: 36.4 ms on one stream, 26.5 ms).  An
// autotuner picks the bucket granularity and, per bucket, the product engine
// (FP64-pipe tiles or the tensor-core kernel) by timing each candidate once on
// the caller's data.
#include <algorithm>
#include <cstring>
#include <map>
#include <new>
#include <vector>

#include "../../include/zolo_csd.h"
#include "solver.h"
#include "tc_gemm.h"

namespace zcsd {

namespace {

constexpr int BATCH_MAX_N = 1024;
constexpr int MAX_LANES = 8;
// Workspace of all lanes together, where more than one needs it: at most this
// much and a quarter of the memory that is free when the plan lays out its
// buckets, so that the caller's later allocations meet the larger part of it.
constexpr size_t LANE_BYTES = (size_t)48 << 30;
constexpr int LANE_FREE_PARTS = 4;
constexpr int BATCH_SWEEPS = 30;  // FP64 Jacobi sweeps at most of a leaf that the refinement leaves open

struct Bucket {
  int nb = 0;                    // padded size
  std::vector<int> inst;         // instance indices
  bool tc = false;               // products on the tensor cores
  int lane = 0;                  // stream and workspace part it runs on
  // device tables (persistent region): per bucket problem p (instance inst[p])
  int* dn = nullptr;             // n_i
  long long* doff = nullptr;     // element offset of instance i in the packed matrices
  long long* dtoff = nullptr;    // offset of instance i in the packed theta
  LeafTable leaves;              // B_p at p nb^2 (ld nb), eigenvalues at p nb
};

// X[2p + w] = diag(A_w of instance p, I), nb x nb (w = 0: A1, 1: A2)
__global__ void pad_gather_kernel(int nb, int P, const int* n, const long long* off, const double* A1,
                                  const double* A2, double* X) {
  const long long nn = (long long)nb * nb;
  const int q = blockIdx.y;
  const int p = q >> 1, w = q & 1, ni = n[p];
  const double* src = (w ? A2 : A1) + off[p];
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nn; t += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(t % nb), c = (int)(t / nb);
    X[q * nn + t] = (r < ni && c < ni) ? src[r + (long long)c * ni] : (r == c ? 1.0 : 0.0);
  }
}

// V_pad[p] = [V_p 0; 0 0] from the packed leaf eigenvectors
__global__ void pad_vectors_kernel(int nb, const int* n, const long long* goff, const double* Vl, double* Vp) {
  const long long nn = (long long)nb * nb;
  const int p = blockIdx.y, ni = n[p];
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nn; t += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(t % nb), c = (int)(t / nb);
    Vp[p * nn + t] = (r < ni && c < ni) ? Vl[goff[p] + r + (long long)c * ni] : 0.0;
  }
}

// One CTA per instance: ascending order of its angles (ties by index), then
// theta, U1, U2, V1 in that column order into the packed outputs; status
// CSD_ERR_NOT_CONVERGED when the instance's Jacobi leaf still rotated in the
// last sweep, CSD_ERR_INTERNAL when an angle is not finite (a failed
// factorization).
__global__ void __launch_bounds__(256) sort_scatter_kernel(int nb, const int* n, const long long* off,
                                                           const long long* toff, const double* th, const double* U1t,
                                                           const double* U2t, const double* Vp, double* theta,
                                                           double* U1, double* U2, double* V1, int* status,
                                                           const int* inst, const int* leaf_done) {
  extern __shared__ double sth[];
  int* rank = (int*)(sth + BATCH_MAX_N);
  const int p = blockIdx.x, ni = n[p];
  const long long nn = (long long)nb * nb;
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int j = threadIdx.x; j < ni; j += blockDim.x) {
    double v = th[(long long)p * nb + j];
    if (!(v == v) || v > 10.0 || v < -10.0) bad = 1;
    sth[j] = v;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < ni; j += blockDim.x) {
    const double v = sth[j];
    int r = 0;
    for (int k = 0; k < ni; ++k) r += (sth[k] < v) || (sth[k] == v && k < j);
    rank[j] = r;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < ni; j += blockDim.x) theta[toff[p] + rank[j]] = sth[j];
  for (long long t = threadIdx.x; t < (long long)ni * ni; t += blockDim.x) {
    const int r = (int)(t % ni), j = (int)(t / ni);
    const long long dst = off[p] + r + (long long)rank[j] * ni, src = p * nn + r + (long long)j * nb;
    U1[dst] = U1t[src];
    U2[dst] = U2t[src];
    V1[dst] = Vp[src];
  }
  if (threadIdx.x == 0) status[inst[p]] = bad ? CSD_ERR_INTERNAL : (leaf_done[p] ? CSD_OK : CSD_ERR_NOT_CONVERGED);
}

}  // namespace

// The product engine of a bucket: the tensor-core kernel or FP64 tiles.
struct EngineScope {
  TcState prev;
  EngineScope(bool tc, Arena& ar, int* err) : prev(t_tc) {
    t_tc = TcState{};
    t_tc.enabled = tc;
    t_tc.sites = ~0u;
    t_tc.ar = &ar;
    t_tc.err = err;
  }
  ~EngineScope() { t_tc = prev; }
};

// One bucket of the batch, enqueued on the context stream with no host
// synchronisation.
void run_bucket(Ctx& cx, Arena& ar, Bucket& bk, const double* A1, const double* A2, double* U1, double* U2, double* V1,
                double* theta, int* status, const int* dinst, int* tc_err) {
  cudaStream_t st = cx.stream;
  const int P = (int)bk.inst.size(), nb = bk.nb;
  const long long nn = (long long)nb * nb;
  const size_t mk = ar.mark();
  EngineScope eng(bk.tc, ar, tc_err);
  double* X = ar.get<double>(2 * P * nn);
  double* W = ar.get<double>(2 * P * nn);
  double* H = ar.get<double>(2 * P * nn);
  double* Bm = ar.get<double>(P * nn);
  double* lam = ar.get<double>((size_t)P * nb);
  double* Vl = ar.get<double>((size_t)bk.leaves.vtot);
  double* Vp = ar.get<double>(P * nn);
  double* T1 = ar.get<double>(P * nn);
  double* T2 = ar.get<double>(P * nn);
  double* C = ar.get<double>((size_t)P * nb);
  double* S = ar.get<double>((size_t)P * nb);
  double* th = ar.get<double>((size_t)P * nb);
  const int gx = (int)std::min<long long>((nn + 255) / 256, 64);
  pad_gather_kernel<<<dim3(gx, 2 * P), 256, 0, st>>>(nb, P, bk.dn, bk.doff, A1, A2, X);
  ZCSD_LAUNCH();
  // lines 1-2 of Algorithm 1 for every block of every instance
  zolo_pd<double>(cx, ar, nb, 2 * P, X, W, nullptr);
  {
    GemmArgs<double> g;  // H = sym(W^* X)
    g.batch = 2 * P;
    g.m = nb; g.n = nb; g.k = nb; g.opA = OP_C; g.opB = OP_N;
    g.A = W; g.lda = nb; g.sA = nn;
    g.B = X; g.ldb = nb; g.sB = nn;
    g.C = H; g.ldc = nb; g.sC = nn;
    g.alpha = 1.0; g.beta = 0.0; g.site = GS_H;
    gemm(g, st);
    symmetrize<double>(st, nb, H, nb, nn, H, nb, nn, 2 * P);
  }
  // line 4: B = H2 - H1 (mu = 0)
  axpby<double>(st, nb, nb, 1.0, H + nn, nb, 2 * nn, 0.0, Bm, nb, nn, P);
  axpby<double>(st, nb, nb, -1.0, H, nb, 2 * nn, 1.0, Bm, nb, nn, P);
  // line 5: every B as one leaf of the batched Jacobi eigensolver
  leaf_solve<double>(cx, ar, bk.leaves, Bm, lam, Vl, BATCH_SWEEPS, true);
  pad_vectors_kernel<<<dim3(gx, P), 256, 0, st>>>(nb, bk.dn, bk.leaves.goff, Vl, Vp);
  ZCSD_LAUNCH();
  // lines 6-9: C, S = diag(V^* H_i V), U_i = W_i V
  auto prod = [&](const double* A, long long sA, double* Cout, int site) {
    GemmArgs<double> g;
    g.batch = P;
    g.m = nb; g.n = nb; g.k = nb; g.opA = OP_N; g.opB = OP_N;
    g.A = A; g.lda = nb; g.sA = sA;
    g.B = Vp; g.ldb = nb; g.sB = nn;
    g.C = Cout; g.ldc = nb; g.sC = nn;
    g.alpha = 1.0; g.beta = 0.0; g.site = site;
    gemm(g, st);
  };
  prod(H, 2 * nn, T1, GS_ASSEMBLY);
  prod(H + nn, 2 * nn, T2, GS_ASSEMBLY);
  col_dots<double>(st, nb, P * nb, Vp, nb, T1, nb, C);
  col_dots<double>(st, nb, P * nb, Vp, nb, T2, nb, S);
  theta_from_cs(st, P * nb, C, S, th);
  prod(W, 2 * nn, T1, GS_ASSEMBLY);       // U1 (padded)
  prod(W + nn, 2 * nn, T2, GS_ASSEMBLY);  // U2 (padded)
  const size_t smem = BATCH_MAX_N * (sizeof(double) + sizeof(int));
  sort_scatter_kernel<<<P, 256, smem, st>>>(nb, bk.dn, bk.doff, bk.dtoff, th, T1, T2, Vp, theta, U1, U2, V1, status,
                                            dinst, bk.leaves.done);
  ZCSD_LAUNCH();
  ar.release(mk);
}

}  // namespace zcsd

using namespace zcsd;

struct csd_batch {
  csd_ctx* owner = nullptr;
  Ctx* cx = nullptr;
  int count = 0;
  std::vector<int> n;
  std::vector<long long> off, toff;
  int gran = 0;                         // chosen bucket granularity
  std::vector<Bucket> buckets;
  char* ws = nullptr;                   // persistent tables + run arena
  size_t ws_bytes = 0, persist_bytes = 0;
  int* dstatus = nullptr;               // per-instance status (device)
  int* dinst = nullptr;                 // bucket-order instance indices (device), per bucket at inst_off
  int* tc_err = nullptr;
  std::vector<int> inst_off;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  const void* bound[6] = {};            // buffers the captured graph reads / writes
  double tune_ms[3] = {0, 0, 0};        // autotuner: batch time per granularity (16, 32, 64)
  bool tuned = false;
  double ws_scale = 1.0;                // grows when a run overflows the arena
  size_t run_need = 0;                  // arena bytes a run was seen to need
  cudaStream_t stream = nullptr;        // the plan's own stream (tuning, capture, replay): lane 0
  cudaEvent_t ev = nullptr;
  int lanes = 1;
  cudaStream_t side[MAX_LANES] = {};    // lanes 1 .. lanes - 1
  cudaStream_t body = nullptr;          // captures the bodies of conditional nodes
  cudaEvent_t side_ev[MAX_LANES] = {};
  size_t lane_off[MAX_LANES + 1] = {};  // workspace parts, from persist_bytes
};

namespace {

size_t bucket_bytes(const Bucket& bk) {
  const long long P = (long long)bk.inst.size(), nb = bk.nb, nn = nb * nb;
  const size_t es = sizeof(double);
  size_t b = (size_t)(2 * P * nn * 3 + P * nn * 4 + P * nb * 4) * es + (size_t)bk.leaves.vtot * 4 * es;
  // zolo_pd on 2P problems plus the tensor-core residues of its largest product
  b += (size_t)(nn * 2 * P * (6 * R_MAX + 6)) * es;
  if (nb >= HOUSEHOLDER_MIN) b += (size_t)(nn * 2 * P * R_MAX) * es;  // the Householder form of the first iteration
  b += tc_gemm_bytes(nb, nb, nb, R_MAX) * 2 * P;
  return b + ((size_t)64 << 20);
}

void free_plan_ws(csd_batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->exec = nullptr;
  b->graph = nullptr;
  if (b->ws) cudaFree(b->ws);
  b->ws = nullptr;
  b->ws_bytes = 0;
}

// Buckets for granularity `gran`, their device tables in the persistent
// region, and the workspace size.
int build_buckets(csd_batch* b, int gran) {
  free_plan_ws(b);
  b->gran = gran;
  std::map<int, std::vector<int>> by;
  for (int i = 0; i < b->count; ++i) by[ceil_div(b->n[i], gran) * gran].push_back(i);
  b->buckets.clear();
  for (auto& kv : by) {
    Bucket bk;
    bk.nb = kv.first;
    bk.inst = kv.second;
    bk.tc = false;
    b->buckets.push_back(bk);
  }
  // persistent region: per bucket n, off, toff and the leaf tables (index
  // arrays, FP32 columns, rotation records); statuses; instance lists; every
  // allocation rounded up to 256 bytes
  size_t pbytes = 0;
  for (auto& bk : b->buckets) {
    std::vector<int> sz;
    for (int i : bk.inst) sz.push_back(b->n[i]);
    pbytes += bk.inst.size() * 128 + leaf_table_bytes(sz, false) + 16 * 256;
  }
  pbytes += (size_t)b->count * 16 + 4 * 256 + (1 << 20);
  std::vector<size_t> need;
  for (auto& bk : b->buckets) {
    long long vt = 0;
    for (int i : bk.inst) vt += (long long)b->n[i] * b->n[i];
    bk.leaves.vtot = vt;
    need.push_back(std::max((size_t)((double)bucket_bytes(bk) * b->ws_scale), b->run_need));
  }
  b->persist_bytes = (pbytes + 255) & ~(size_t)255;
  // lanes: the largest buckets first, each to the lane with the least work so
  // far (a bucket's time grows with its size, hardly with its instances); as
  // many lanes as fit the limit (one lane needs no more than the largest bucket)
  size_t free_bytes = 0, device_bytes = 0;
  if (cudaMemGetInfo(&free_bytes, &device_bytes) != cudaSuccess) cudaGetLastError();
  const size_t limit = std::min(LANE_BYTES, free_bytes / LANE_FREE_PARTS);
  std::vector<int> order((int)b->buckets.size());
  for (size_t k = 0; k < order.size(); ++k) order[k] = (int)k;
  std::sort(order.begin(), order.end(), [&](int x, int y) { return b->buckets[x].nb > b->buckets[y].nb; });
  for (b->lanes = std::min<int>(MAX_LANES, (int)b->buckets.size());; --b->lanes) {
    size_t bytes[MAX_LANES] = {}, total = 0;
    double load[MAX_LANES] = {};
    for (int k : order) {
      const int l = (int)(std::min_element(load, load + b->lanes) - load);
      b->buckets[k].lane = l;
      load[l] += b->buckets[k].nb + 32.0;
      bytes[l] = std::max(bytes[l], (need[k] + 255) & ~(size_t)255);
    }
    for (int l = 0; l < b->lanes; ++l) {
      b->lane_off[l] = total;
      total += bytes[l];
    }
    b->lane_off[b->lanes] = total;
    if (b->lanes > 1 && total > limit) continue;
    b->ws_bytes = b->persist_bytes + total;
    if (cudaMalloc((void**)&b->ws, b->ws_bytes) == cudaSuccess) break;
    cudaGetLastError();
    b->ws = nullptr;
    b->ws_bytes = 0;
    if (b->lanes == 1) return CSD_ERR_ALLOC;
  }
  Ctx& cx = *b->cx;
  Arena per;
  per.base = b->ws;
  per.cap = b->persist_bytes;
  try {
    b->dstatus = per.get<int>(b->count);
    b->tc_err = per.get<int>(1);
    b->dinst = per.get<int>(b->count);
    b->inst_off.clear();
    std::vector<int> all;
    for (auto& bk : b->buckets) {
      b->inst_off.push_back((int)all.size());
      all.insert(all.end(), bk.inst.begin(), bk.inst.end());
      const int P = (int)bk.inst.size();
      std::vector<int> hn(P);
      std::vector<long long> ho(P), ht(P), boff(P);
      std::vector<int> lds(P, bk.nb), loff(P);
      for (int p = 0; p < P; ++p) {
        const int i = bk.inst[p];
        hn[p] = b->n[i];
        ho[p] = b->off[i];
        ht[p] = b->toff[i];
        boff[p] = (long long)p * bk.nb * bk.nb;
        loff[p] = p * bk.nb;
      }
      bk.dn = per.get<int>(P);
      bk.doff = per.get<long long>(P);
      bk.dtoff = per.get<long long>(P);
      ZCSD_CUDA(cudaMemcpyAsync(bk.dn, hn.data(), sizeof(int) * P, cudaMemcpyHostToDevice, cx.stream));
      ZCSD_CUDA(cudaMemcpyAsync(bk.doff, ho.data(), sizeof(long long) * P, cudaMemcpyHostToDevice, cx.stream));
      ZCSD_CUDA(cudaMemcpyAsync(bk.dtoff, ht.data(), sizeof(long long) * P, cudaMemcpyHostToDevice, cx.stream));
      bk.leaves = leaf_table_build(cx, per, boff, lds, loff, hn, false);
    }
    ZCSD_CUDA(cudaMemcpyAsync(b->dinst, all.data(), sizeof(int) * b->count, cudaMemcpyHostToDevice, cx.stream));
    ZCSD_CUDA(cudaStreamSynchronize(cx.stream));
  } catch (ArenaOverflow&) {
    return CSD_ERR_INTERNAL;
  } catch (CudaFail&) {
    return CSD_ERR_CUDA;
  }
  return CSD_OK;
}

struct StreamSwap {
  Ctx& c;
  cudaStream_t prev;
  StreamSwap(Ctx& c_, cudaStream_t s) : c(c_), prev(c_.stream) { c.stream = s; }
  ~StreamSwap() { c.stream = prev; }
};

// The whole batch, forked from and joined to the context stream (capturable:
// no host sync).
void run_all(csd_batch* b, const double* A1, const double* A2, double* U1, double* U2, double* V1, double* theta) {
  Ctx& cx = *b->cx;
  ZCSD_CUDA(cudaEventRecord(b->ev, cx.stream));
  for (int l = 1; l < b->lanes; ++l) ZCSD_CUDA(cudaStreamWaitEvent(b->side[l], b->ev, 0));
  for (int l = 0; l < b->lanes; ++l) {
    StreamSwap lane(cx, l ? b->side[l] : cx.stream);
    for (size_t k = 0; k < b->buckets.size(); ++k) {
      if (b->buckets[k].lane != l) continue;
      Arena ar;
      ar.base = b->ws + b->persist_bytes + b->lane_off[l];
      ar.cap = b->lane_off[l + 1] - b->lane_off[l];
      run_bucket(cx, ar, b->buckets[k], A1, A2, U1, U2, V1, theta, b->dstatus, b->dinst + b->inst_off[k], b->tc_err);
    }
  }
  for (int l = 1; l < b->lanes; ++l) {
    ZCSD_CUDA(cudaEventRecord(b->side_ev[l], b->side[l]));
    ZCSD_CUDA(cudaStreamWaitEvent(cx.stream, b->side_ev[l], 0));
  }
}

// The whole batch as a graph (b->graph, b->exec) bound to the caller's buffers.
void capture_all(csd_batch* b, const double* A1, const double* A2, double* U1, double* U2, double* V1, double* theta) {
  Ctx& cx = *b->cx;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->exec = nullptr;
  b->graph = nullptr;
  ZCSD_CUDA(cudaStreamBeginCapture(cx.stream, cudaStreamCaptureModeThreadLocal));
  run_all(b, A1, A2, U1, U2, V1, theta);
  ZCSD_CUDA(cudaStreamEndCapture(cx.stream, &b->graph));
  ZCSD_CUDA(cudaGraphInstantiate(&b->exec, b->graph, 0));
  const void* bound[6] = {A1, A2, U1, U2, V1, theta};
  std::memcpy(b->bound, bound, sizeof(bound));
}

// After a failure inside a capture: leaves the streams uncaptured.
void end_captures(csd_batch* b) {
  cudaStreamCaptureStatus cs;
  cudaGraph_t g = nullptr;
  // a body's graph belongs to the conditional node of the outer one
  if (cudaStreamIsCapturing(b->body, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone)
    cudaStreamEndCapture(b->body, &g);
  g = nullptr;
  if (cudaStreamIsCapturing(b->stream, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
    cudaStreamEndCapture(b->stream, &g);
    if (g) cudaGraphDestroy(g);
  }
}

// Per bucket engine choice (each bucket alone), then the granularity whose
// whole batch is fastest, buckets side by side as in a later run (the sum over
// the buckets alone counts the small ones that others hide: 48 instances of
// 16..256 rows took granularity 64, 27.6 ms, over 16, 25.6 ms).  The finest
// comes last, is the usual choice and then keeps its graph.
int autotune(csd_batch* b, const double* A1, const double* A2, double* U1, double* U2, double* V1, double* theta) {
  const int grans[3] = {16, 32, 64};
  double best_total = 1e300;
  int best_g = 32;
  std::vector<char> best_tc;
  for (int gi = 2; gi >= 0; --gi) {
    int st = build_buckets(b, grans[gi]);
    if (st) return st;
    std::vector<char> choice;
    Ctx& cx = *b->cx;
    cudaEvent_t e0, e1;
    for (auto& bk : b->buckets) {
      Arena ar;
      ar.base = b->ws + b->persist_bytes;
      ar.cap = b->ws_bytes - b->persist_bytes;
      float ms[2];
      for (int e = 0; e < 2; ++e) {
        bk.tc = e == 1;
        const int* dinst = b->dinst + b->inst_off[&bk - &b->buckets[0]];
        run_bucket(cx, ar, bk, A1, A2, U1, U2, V1, theta, b->dstatus, dinst, b->tc_err);  // warm
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        cudaEventRecord(e0, cx.stream);
        run_bucket(cx, ar, bk, A1, A2, U1, U2, V1, theta, b->dstatus, dinst, b->tc_err);
        cudaEventRecord(e1, cx.stream);
        ZCSD_CUDA(cudaEventSynchronize(e1));
        cudaEventElapsedTime(&ms[e], e0, e1);
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
      }
      bk.tc = ms[1] < ms[0];
      choice.push_back(bk.tc);
    }
    capture_all(b, A1, A2, U1, U2, V1, theta);
    ZCSD_CUDA(cudaGraphUpload(b->exec, cx.stream));
    float total = 0.0f;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, cx.stream);
    ZCSD_CUDA(cudaGraphLaunch(b->exec, cx.stream));
    cudaEventRecord(e1, cx.stream);
    ZCSD_CUDA(cudaEventSynchronize(e1));
    cudaEventElapsedTime(&total, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->tune_ms[gi] = total;
    if (total < best_total) {
      best_total = total;
      best_g = grans[gi];
      best_tc = choice;
    }
  }
  if (b->gran != best_g) {
    int st = build_buckets(b, best_g);
    if (st) return st;
    for (size_t k = 0; k < b->buckets.size(); ++k) b->buckets[k].tc = best_tc[k];
  }
  b->tuned = true;
  return CSD_OK;
}

}  // namespace


// Access to the context behind the opaque handle (solver.cu defines it).
zcsd::Ctx* ctx_internal(csd_ctx* ctx);

int csd_batch_create(csd_ctx* ctx, int count, const int* n, csd_batch** plan) {
  if (!ctx) return -1;
  if (count < 1) return -2;
  if (!n) return -3;
  if (!plan) return -4;
  for (int i = 0; i < count; ++i)
    if (n[i] < 1 || n[i] > BATCH_MAX_N) return -3;
  csd_batch* b = new (std::nothrow) csd_batch();
  if (!b) return CSD_ERR_ALLOC;
  b->owner = ctx;
  b->cx = ctx_internal(ctx);
  b->count = count;
  b->n.assign(n, n + count);
  b->off.assign(count + 1, 0);
  b->toff.assign(count + 1, 0);
  for (int i = 0; i < count; ++i) {
    b->off[i + 1] = b->off[i] + (long long)n[i] * n[i];
    b->toff[i + 1] = b->toff[i] + n[i];
  }
  *plan = b;
  return CSD_OK;
}

int csd_batch_run(csd_batch* b, const double* A1, const double* A2, double* U1, double* U2, double* V1,
                  double* theta, int* status) {
  if (!b) return -1;
  if (!A1) return -2;
  if (!A2) return -3;
  if (!U1) return -4;
  if (!U2) return -5;
  if (!V1) return -6;
  if (!theta) return -7;
  Ctx& cx = *b->cx;
  if (cudaSetDevice(cx.device) != cudaSuccess) {
    cudaGetLastError();
    return CSD_ERR_CUDA;
  }
  struct ProfOff {
    Profiler* prev;
    ProfOff() : prev(t_prof) { t_prof = nullptr; }
    ~ProfOff() { t_prof = prev; }
  } prof_off;
  // the batch runs on the plan's own non-blocking stream (a capture needs a
  // stream other than the legacy default one), ordered after the work
  // already queued on the context's stream and before whatever follows it
  if (!b->stream) {
    bool ok = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&b->ev, cudaEventDisableTiming) == cudaSuccess &&
              cudaStreamCreateWithFlags(&b->body, cudaStreamNonBlocking) == cudaSuccess;
    for (int l = 1; l < MAX_LANES; ++l)
      ok = ok && cudaStreamCreateWithFlags(&b->side[l], cudaStreamNonBlocking) == cudaSuccess &&
           cudaEventCreateWithFlags(&b->side_ev[l], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
      cudaGetLastError();
      return CSD_ERR_CUDA;
    }
  }
  if (cudaEventRecord(b->ev, cx.stream) != cudaSuccess || cudaStreamWaitEvent(b->stream, b->ev, 0) != cudaSuccess) {
    cudaGetLastError();
    return CSD_ERR_CUDA;
  }
  StreamSwap swap(cx, b->stream);
  cx.body_stream = b->body;
  for (int attempt = 0;; ++attempt) {
   try {
    if (!b->tuned) {
      const int st = autotune(b, A1, A2, U1, U2, V1, theta);
      if (st) return st;
    }
    const void* want[6] = {A1, A2, U1, U2, V1, theta};
    if (!b->exec || std::memcmp(want, b->bound, sizeof(want)) != 0) {
      ZCSD_CUDA(cudaMemsetAsync(b->tc_err, 0, sizeof(int), cx.stream));
      run_all(b, A1, A2, U1, U2, V1, theta);  // uncaptured once: lazy set-up outside the capture
      ZCSD_CUDA(cudaStreamSynchronize(cx.stream));
      capture_all(b, A1, A2, U1, U2, V1, theta);
    }
    ZCSD_CUDA(cudaMemsetAsync(b->tc_err, 0, sizeof(int), cx.stream));
    ZCSD_CUDA(cudaGraphLaunch(b->exec, cx.stream));
    ZCSD_CUDA(cudaStreamSynchronize(cx.stream));
    int err = 0;
    ZCSD_CUDA(cudaMemcpy(&err, b->tc_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (status) ZCSD_CUDA(cudaMemcpy(status, b->dstatus, sizeof(int) * b->count, cudaMemcpyDeviceToHost));
    if (err) return CSD_ERR_DEVICE_TIMEOUT;
    return CSD_OK;
   } catch (ArenaOverflow& o) {
    // a run needed more workspace than estimated: grow it and redo the set-up
    end_captures(b);
    cudaStreamSynchronize(cx.stream);
    for (int l = 1; l < MAX_LANES; ++l) cudaStreamSynchronize(b->side[l]);
    cudaGetLastError();
    if (attempt >= 6) return CSD_ERR_INTERNAL;
    b->ws_scale *= 2.0;
    b->run_need = std::max(b->run_need, o.needed + o.needed / 4);
    std::vector<char> tcs;
    for (auto& bk : b->buckets) tcs.push_back(bk.tc);
    const bool tuned = b->tuned;
    const int st = build_buckets(b, b->gran ? b->gran : 32);
    if (st) return st;
    for (size_t k = 0; k < b->buckets.size() && k < tcs.size(); ++k) b->buckets[k].tc = tcs[k];
    b->tuned = tuned;
    std::memset(b->bound, 0, sizeof(b->bound));
    continue;
   } catch (CudaFail& f) {
    fprintf(stderr, "zolo_csd: CUDA error %s at %s:%d\n", cudaGetErrorString(f.err), f.file, f.line);
    end_captures(b);
    cudaGetLastError();
    return CSD_ERR_CUDA;
   }
  }
}

int csd_batch_destroy(csd_batch* b) {
  if (!b) return CSD_OK;
  cudaSetDevice(b->cx->device);
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (int l = 1; l < MAX_LANES; ++l) {
    if (b->side[l]) {
      cudaStreamSynchronize(b->side[l]);
      cudaStreamDestroy(b->side[l]);
    }
    if (b->side_ev[l]) cudaEventDestroy(b->side_ev[l]);
  }
  free_plan_ws(b);
  if (b->body) cudaStreamDestroy(b->body);
  if (b->ev) cudaEventDestroy(b->ev);
  if (b->stream) cudaStreamDestroy(b->stream);
  delete b;
  return CSD_OK;
}

int csd_batch_stats(const csd_batch* b, int* granularity, int* buckets, int* tc_buckets, double* tune_ms) {
  if (!b) return -1;
  if (granularity) *granularity = b->gran;
  if (buckets) *buckets = (int)b->buckets.size();
  if (tc_buckets) {
    int c = 0;
    for (auto& bk : b->buckets) c += bk.tc;
    *tc_buckets = c;
  }
  if (tune_ms)
    for (int i = 0; i < 3; ++i) tune_ms[i] = b->tune_ms[i];
  return CSD_OK;
}
