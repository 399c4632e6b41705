// FP64-accurate GEMM on the tcgen05 tensor cores by residue arithmetic
// (tc_gemm.cu).  Real FP64 only; op(A), op(B) in {N, T}.
#pragma once
#include "linalg.h"

namespace zcsd {

// Per-call tensor-core state of the running entry point (thread-local): when
// `enabled`, gemm<double>() sends eligible products to tc_gemm() using this
// arena and error flag.
struct TcState {
  bool enabled = false;
  unsigned sites = 0;  // bit s: GEMM call site s (GemmSite) may run on the tensor cores
  Arena* ar = nullptr;
  int* err = nullptr;
  long long probe_wait = 0;  // > 0: each launch first polls a barrier nothing signals (timeout-path tests)
  int flush_every = 0;       // > 0: drains between reductions of the running residue sums (tests of that path)
  unsigned reduced_sites = 0;  // bit s: call site s keeps reduced_bits bits of an operand instead of 56
  int reduced_bits = 56;
};
extern thread_local TcState t_tc;
// true when gemm<double>(g) will run on the tensor cores
bool tc_will_handle(const GemmArgs<double>& g);
// C = alpha sum_j w_j op(A_j) op(B_j) + beta Cin, as gemm() (ksplit = 1);
// workspace comes from `ar`; *err is set to 1 if a tensor-core wait timed out.
void tc_gemm(const GemmArgs<double>& g, cudaStream_t st, Arena& ar, int* err);
// workspace bytes of an m x n product over nsum terms of k, at most
size_t tc_gemm_bytes(long long m, long long n, long long k, int nsum);

// Complex FP64 products with real alpha and beta as two real grouped sums
// over the interleaved real and imaginary parts (element stride 2):
// Re C = Re A Re B - Im A Im B, Im C = Re A Im B + Im A Re B (signs of the
// conjugate transposes folded into the term weights).
bool tc_will_handle_complex(const GemmArgs<z64>& g);
void tc_gemm_complex(const GemmArgs<z64>& g, cudaStream_t st, Arena& ar, int* err);

}  // namespace zcsd
