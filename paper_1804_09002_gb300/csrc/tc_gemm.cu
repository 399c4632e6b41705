// FP64-accurate GEMM on the tcgen05 tensor cores (sm_103a) by residue number
// systems (the Ozaki scheme II: Ozaki, Uchino and Imamura, "Ozaki Scheme II: A
// GEMM-oriented emulation of floating-point matrix multiplication using an
// integer modular technique", 2025).
//
// Every row i of op(A) is scaled by 2^(beta - ea_i) (ea_i = exponent of the
// row's largest |entry|, shared by all terms of a grouped sum) and rounded to
// an integer of magnitude at most 2^beta, beta = 56; likewise every column j of
// op(B).  The integer product, below P / 2 for P = p_1 ... p_s the product of
// s pairwise coprime moduli of about 9 bits, follows from its residues: s
// products of the operands' balanced residues, |r| <= 256, which are exact in
// BF16.  256 consecutive terms of such a product stay within 2^24, exact in
// the FP32 accumulators.  s = 14 for up to 4096 terms: half of the 28 products
// that eight-bit slices need for the same 56 bits, each one an ordinary GEMM
// with one accumulator instead of seven.
//
// Four launches:
//  * tc_exp_kernel: row exponents; tc_convert_kernel: integers and residues,
//    stored as 128-row x
//    64-k chunks of 16 KiB per modulus in the order in which the tensor cores
//    read shared memory (K-major rows of 128 bytes, 128-byte swizzle; two
//    chunks in a row are 256 rows);
//  * tc_gemm_kernel: persistent, one CTA per SM over items (128 x 256 output
//    tile, modulus, problem).  One warp copies 64-k stages into a ring of
//    four with cp.async.bulk; one lane issues M = 128, N = 256, K = 16 MMAs;
//    sixteen epilogue warps reduce the accumulators mod p every 256 k while
//    the next 256 accumulate in the other half of TMEM, and store the residue
//    of (product x weight of the modulus) as 16-bit integers;
//  * tc_combine_kernel: the Chinese remainder sum as a 96-bit fixed-point
//    fraction of P, its sign and scale, alpha and beta C.
// Every wait is bounded; a wait that runs out sets the CTA's abort flag and
// the device error flag, every role leaves its loop, the producer waits
// (bounded) for its copies in flight and the MMA issuer for its MMAs before
// TMEM is released, and the combining kernel then writes NaN.
#include <cuda_bf16.h>

#include <climits>
#include <mutex>

#include "tc_gemm.h"

namespace zcsd {

namespace {

constexpr int TC_BM = 128, TC_BN = 256, TC_BK = 64;
constexpr int TC_CHUNK = TC_BM * TC_BK;  // elements of a stored chunk (16 KiB)
constexpr int TC_NSTAGE = 4;
constexpr int TC_A_STAGE = TC_BM * TC_BK * 2;
constexpr int TC_STAGE = TC_A_STAGE + TC_BN * TC_BK * 2;
constexpr int TC_SMEM = TC_NSTAGE * TC_STAGE + 1024;
constexpr int TC_DRAIN = 256 / TC_BK;  // stages between reductions of an accumulator
constexpr int TC_FOLD = 32768;  // drains between reductions of their sum: 257 x 32769 < 2^24 stays exact in FP32
constexpr int TC_EPI_WARPS = 16;
constexpr int TC_THREADS = 32 * (2 + TC_EPI_WARPS);
constexpr int TC_CPT = TC_BN / 4;  // accumulator columns per epilogue thread
constexpr long long TC_WAIT_LIMIT = 1LL << 26;
constexpr int TC_MAXMOD = 16;

// Pairwise coprime moduli with balanced residues of at most 255 (254 for the
// even one): the largest such set below 512, greedily.
constexpr int TC_MODULI[TC_MAXMOD] = {511, 509, 508, 507, 505, 503, 499, 493, 491, 487, 479, 473, 467, 463, 461, 457};

// Constants of a product with nmod moduli.
struct RnsTab {
  int nmod, bits;
  float p[TC_MAXMOD], inv[TC_MAXMOD];       // modulus and its reciprocal
  float c1[TC_MAXMOD], c2[TC_MAXMOD], c3[TC_MAXMOD];  // 2^14, 2^28, 2^42 mod p, balanced
  float q[TC_MAXMOD];                       // (P / p)^-1 mod p, balanced
  unsigned C0[TC_MAXMOD], C1[TC_MAXMOD], C2[TC_MAXMOD];  // round(2^96 / p), 32-bit words
  unsigned long long Pm;                    // P = Pm 2^Pe to 64 bits, bit 63 set
  int Pe;
  double log2P;
};

int mod_inverse(int a, int p) {
  for (int x = 1; x < p; ++x)
    if ((long long)a * x % p == 1) return x;
  return 1;
}

RnsTab make_tab(int nmod) {
  RnsTab t{};
  t.nmod = nmod;
  unsigned long long w[4] = {1, 0, 0, 0};  // P, 256 bits little-endian
  for (int i = 0; i < nmod; ++i) {
    const int p = TC_MODULI[i];
    auto bal = [p](long long v) {
      int r = (int)(((v % p) + p) % p);
      return (float)(r > p / 2 ? r - p : r);
    };
    t.p[i] = (float)p;
    t.inv[i] = 1.0f / (float)p;
    t.c1[i] = bal(1LL << 14);
    t.c2[i] = bal(1LL << 28);
    t.c3[i] = bal(1LL << 42);
    int rest = 1;
    for (int k = 0; k < nmod; ++k)
      if (k != i) rest = rest * TC_MODULI[k] % p;
    t.q[i] = bal(mod_inverse(rest, p));
    const unsigned __int128 two96 = (unsigned __int128)1 << 96;
    const unsigned __int128 C = (two96 + p / 2) / p;
    t.C0[i] = (unsigned)C;
    t.C1[i] = (unsigned)(C >> 32);
    t.C2[i] = (unsigned)(C >> 64);
    unsigned __int128 carry = 0;
    for (int k = 0; k < 4; ++k) {
      const unsigned __int128 v = (unsigned __int128)w[k] * p + carry;
      w[k] = (unsigned long long)v;
      carry = v >> 64;
    }
    t.log2P += std::log2((double)p);
  }
  int top = 3;
  while (top > 0 && !w[top]) --top;
  const int lz = __builtin_clzll(w[top]);
  t.Pm = w[top] << lz;
  if (lz && top > 0) t.Pm |= w[top - 1] >> (64 - lz);
  t.Pe = 64 * top - lz;
  return t;
}

// Fewest moduli that hold a sum of K products of bits-bit integers.
const RnsTab& pick_tab(int bits, double K) {
  static RnsTab tabs[TC_MAXMOD + 1];
  static std::once_flag once;
  std::call_once(once, [] {
    for (int i = 1; i <= TC_MAXMOD; ++i) tabs[i] = make_tab(i);
  });
  const double need = 2.0 * bits + 1.0 + std::log2(std::max(K, 1.0)) + 0.01;
  for (int i = 1; i < TC_MAXMOD; ++i)
    if (tabs[i].log2P >= need) return tabs[i];
  return tabs[TC_MAXMOD];
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// tcgen05 shared-memory matrix descriptor of K-major rows of 128 bytes in the
// 128-byte swizzle (16-byte unit c of row r at unit c ^ (r mod 8)): start
// address, 1024 bytes between 8-row groups, descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t add) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(ad), "l"(bd), "r"(idesc), "r"(add));
}

// arrive on `mbar` when the MMAs issued so far are done
__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t addr, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count));
}

__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(addr), "r"(parity)
      : "memory");
  return done != 0;
}

// Bounded wait for the phase of `parity`; gives up after `limit` polls or
// as soon as the CTA's abort flag is set.  Returns true on completion.
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity, volatile int* abort_flag,
                                          long long limit = TC_WAIT_LIMIT) {
  for (long long it = 0; it < limit; ++it) {
    if (mbar_try(addr, parity)) return true;
    if (abort_flag && *abort_flag) return false;
  }
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t addr) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(addr) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t addr, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr), "r"(bytes) : "memory");
}

// contiguous copy into shared memory (both sides 16-byte aligned, a multiple
// of 16 bytes), completion counted on `mbar`
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"((uint64_t)__cvta_generic_to_global(src)), "r"(bytes), "r"(mbar)
               : "memory");
}

// 16 columns of this warp's TMEM lanes, on their way until tmem_wait16 has
// returned (which names the registers, so that nothing reads them before)
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
}
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// two FP32 lanes in one register pair
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// v - round(v / p) p per lane for integers |v| <= 2^24 (|result| <= p / 2 + 1),
// exact; np = -p, magic = 1.5 2^23 (adding it rounds to an integer)
__device__ __forceinline__ f32x2 mod_p2(f32x2 v, f32x2 np, f32x2 inv, f32x2 magic, f32x2 nmagic) {
  const f32x2 q = add2(fma2(v, inv, magic), nmagic);
  return fma2(q, np, v);
}

// J 2^e as a double, rounded to nearest (ties to even on J's bits), built with
// integer instructions: GB300's FP64 pipe retires 2 lanes per clock per SM.
// Results outside the normal range take ldexp.
__device__ __forceinline__ double mag_to_double(unsigned long long m, int e, unsigned long long sgn) {
  // m: bit 63 set; value m 2^e
  unsigned long long mant = m >> 11;  // 53 bits with the leading one
  const unsigned long long rem = m & 0x7FFull;
  int E = 63 + e;
  if (rem > 0x400ull || (rem == 0x400ull && (mant & 1ull))) {
    ++mant;
    if (mant >> 53) {
      mant >>= 1;
      ++E;
    }
  }
  if (E < -1022 || E > 1023) {
    const double v = ldexp((double)mant, E - 52);
    return sgn ? -v : v;
  }
  return __longlong_as_double((long long)(sgn | ((unsigned long long)(E + 1023) << 52) | (mant & 0xFFFFFFFFFFFFFull)));
}

struct TcArgs {
  int m, n, kpad, nsum;
  int nrbA, nrbB, nkb;       // 128-row blocks of the operands, 64-k blocks
  int batch, bstrideA, bstrideB;  // problems; 0: all problems share that operand
  int kb_flags, uplo, nmod;
  int fold;                  // drains between reductions of the running sum (TC_FOLD at most)
  int tiles_m, tiles_n, tiles;  // output tiles, and those that uplo keeps (per problem and modulus)
  const __nv_bfloat16 *A, *B;
  unsigned short* R;         // [problem][modulus][n][128 tiles_m] residues
  int* err;
  long long probe_wait;      // > 0: first poll a barrier nothing signals (timeout-path tests)
};

// One item: an output tile of one problem and modulus, with its 64-k stages.
struct TcItem {
  int mt, nt, z, mod, kb0, nst;
};

__host__ __device__ inline int tile_rows(int uplo, int nt, int tiles_m) {
  // tiles of column block nt that touch the upper triangle (uplo 1): m0 <= n0 + 255
  return uplo == 1 ? (2 * (nt + 1) < tiles_m ? 2 * (nt + 1) : tiles_m) : tiles_m;
}

__device__ __forceinline__ TcItem tc_item(const TcArgs& g, long long it) {
  TcItem t;
  const int per = g.tiles;
  int r = (int)(it % per);
  const long long zm = it / per;
  t.mod = (int)(zm % g.nmod);
  t.z = (int)(zm / g.nmod);
  if (g.uplo == 1) {
    t.nt = 0;
    for (int c; r >= (c = tile_rows(1, t.nt, g.tiles_m)); ++t.nt) r -= c;
    t.mt = r;
  } else {
    t.mt = r % g.tiles_m;
    t.nt = r / g.tiles_m;
  }
  int kb = 0, ke = g.kpad;
  const int m0 = t.mt * TC_BM, n0 = t.nt * TC_BN;
  if (g.kb_flags & K_FROM_COL) kb = max(kb, n0);
  if (g.kb_flags & K_FROM_ROW) kb = max(kb, m0);
  if (g.kb_flags & K_TO_COL) ke = min(ke, n0 + TC_BN);
  if (g.kb_flags & K_TO_ROW) ke = min(ke, m0 + TC_BM);
  t.kb0 = kb / TC_BK;
  t.nst = ke > kb ? (ke - t.kb0 * TC_BK + TC_BK - 1) / TC_BK : 0;
  return t;
}

// FOLD: some item has more drains than g.fold, so its running sum is reduced on
// the way (the others' code is without it).
template <bool FOLD>
__global__ void __launch_bounds__(TC_THREADS, 1) tc_gemm_kernel(const TcArgs g, const __grid_constant__ RnsTab tab) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full_bar[TC_NSTAGE], empty_bar[TC_NSTAGE];
  __shared__ __align__(8) uint64_t accf_bar[2], acce_bar[2], done_bar, probe_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  volatile int* abort_v = &abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long items = (long long)g.tiles * g.nmod * g.batch;

  if (tid == 0) {
    for (int i = 0; i < TC_NSTAGE; ++i) {
      mbar_init(smem_u32(&full_bar[i]), 1);
      mbar_init(smem_u32(&empty_bar[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&accf_bar[i]), 1);
      mbar_init(smem_u32(&acce_bar[i]), TC_EPI_WARPS);
    }
    mbar_init(smem_u32(&done_bar), 1);
    mbar_init(smem_u32(&probe_bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  auto fail = [&]() {
    *abort_v = 1;
    atomicExch(g.err, 1);
  };

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0 && g.probe_wait > 0 && !mbar_wait(smem_u32(&probe_bar), 0u, abort_v, g.probe_wait)) fail();
    __syncwarp();
    // slots and phases are counted, not divided out: a stage lasts 512 clocks,
    // and one lane's address arithmetic was what set the pace before
    int slot = 0, issued = 0;
    uint32_t phase = 1;
    bool ok = __shfl_sync(0xffffffffu, *abort_v, 0) == 0;  // one lane's view: the loop is warp-uniform
    for (long long it = blockIdx.x; it < items && ok; it += gridDim.x) {
      const TcItem t = tc_item(g, it);
      // lane 0: A's chunks; lanes 1, 2: B's
      const int rb = lane == 0 ? t.mt : min(2 * t.nt + lane - 1, g.nrbB - 1);
      const int nrb = lane == 0 ? g.nrbA : g.nrbB, zs = lane == 0 ? g.bstrideA : g.bstrideB;
      for (int js = 0; js < g.nsum && ok; ++js) {
        const __nv_bfloat16* src =
            (lane == 0 ? g.A : g.B) +
            ((((long long)(t.z * zs * g.nsum + js) * nrb + rb) * g.nmod + t.mod) * g.nkb + t.kb0) * TC_CHUNK;
        for (int q = 0; q < t.nst; ++q, src += TC_CHUNK) {
          const uint32_t fb = smem_u32(&full_bar[slot]);
          int go = 1;
          if (lane == 0) {
            go = mbar_wait(smem_u32(&empty_bar[slot]), phase, abort_v);
            if (!go && !*abort_v) fail();
            if (go) mbar_expect_tx(fb, TC_STAGE);
          }
          ok = __shfl_sync(0xffffffffu, go, 0) != 0;
          if (!ok) break;
          if (lane < 3)
            bulk_load(smem_u32(smem + slot * TC_STAGE) + lane * (TC_CHUNK * 2), src, TC_CHUNK * 2, fb);
          issued = min(issued + 1, TC_NSTAGE);
          if (++slot == TC_NSTAGE) {
            slot = 0;
            phase ^= 1;
          }
        }
      }
    }
    // no copy may still be writing shared memory when the CTA exits: the
    // last stages issued (at most one per slot) must have landed
    if (lane == 0)
      for (; issued > 0; --issued) {
        if (--slot < 0) {
          slot = TC_NSTAGE - 1;
          phase ^= 1;
        }
        if (!mbar_wait(smem_u32(&full_bar[slot]), phase ^ 1, nullptr)) fail();
      }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int slot = 0;
      uint32_t phase = 0;
      unsigned cycle = 0;  // drains issued: accumulator half cycle & 1
      const uint64_t desc0 = smem_desc(smem_u32(smem));
      bool ok = true;
      for (long long it = blockIdx.x; it < items && ok && !*abort_v; it += gridDim.x) {
        const TcItem t = tc_item(g, it);
        const int Q = g.nsum * t.nst;
        for (int q = 0; q < Q && ok; ++cycle) {
          const uint32_t acc = tmem + (cycle & 1u) * TC_BN;
          if (!mbar_wait(smem_u32(&acce_bar[cycle & 1u]), ((cycle >> 1) & 1u) ^ 1u, abort_v)) {
            if (!*abort_v) fail();
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const int q1 = min(Q, q + TC_DRAIN);
          for (int f = q; f < q1; ++f) {
            if (!mbar_wait(smem_u32(&full_bar[slot]), phase, abort_v)) {
              if (!*abort_v) fail();
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t da = desc0 + (uint64_t)(slot * (TC_STAGE >> 4)), db = da + (TC_A_STAGE >> 4);
#pragma unroll
            for (int ks = 0; ks < TC_BK / 16; ++ks)
              mma_bf16(acc, da + 2 * ks, db + 2 * ks, idesc_bf16(TC_BM, TC_BN), (f > q || ks > 0) ? 1u : 0u);
            mma_commit(smem_u32(&empty_bar[slot]));
            if (++slot == TC_NSTAGE) {
              slot = 0;
              phase ^= 1;
            }
          }
          if (!ok) break;
          mma_commit(smem_u32(&accf_bar[cycle & 1u]));
          q = q1;
        }
      }
      // every MMA issued has completed before TMEM is released
      mma_commit(smem_u32(&done_bar));
      if (!mbar_wait(smem_u32(&done_bar), 0u, nullptr)) fail();
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int lq = warp & 3, ch = (warp - 2) >> 2;  // TMEM lane quarter, column quarter
    const uint32_t tmem_row = tmem + ((uint32_t)(32 * lq) << 16) + (uint32_t)(TC_CPT * ch);
    const int ldr = TC_BM * g.tiles_m;
    unsigned cycle = 0;
    bool ok = true;
    for (long long it = blockIdx.x; it < items && ok; it += gridDim.x) {
      const TcItem t = tc_item(g, it);
      const int Q = g.nsum * t.nst;
      const float p = tab.p[t.mod], inv = tab.inv[t.mod];
      const f32x2 np2 = pack2(-p, -p), inv2 = pack2(inv, inv), mg2 = pack2(12582912.0f, 12582912.0f),
                  nmg2 = pack2(-12582912.0f, -12582912.0f);
      f32x2 acc[TC_CPT / 2];
#pragma unroll
      for (int c = 0; c < TC_CPT / 2; ++c) acc[c] = 0ull;
      int left = g.fold;
      for (int q = 0; q < Q; q += TC_DRAIN, ++cycle) {
        // uniform over the warp: the TMEM accesses below are warp-collective
        ok = __all_sync(0xffffffffu, !*abort_v && mbar_wait(smem_u32(&accf_bar[cycle & 1u]), (cycle >> 1) & 1u, abort_v));
        if (!ok) {
          if (!*abort_v) fail();
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        // the next 16 columns are on their way while these are reduced
        uint32_t r[2][16];
        const uint32_t base = tmem_row + (cycle & 1u) * TC_BN;
        tmem_ld16(base, r[0]);
#pragma unroll
        for (int h = 0; h < TC_CPT / 16; ++h) {
          tmem_wait16(r[h & 1]);
          if (h + 1 < TC_CPT / 16) {
            tmem_ld16(base + 16 * (h + 1), r[(h + 1) & 1]);
          } else {  // read out: the MMAs may overwrite this half
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acce_bar[cycle & 1u]));
          }
#pragma unroll
          for (int c = 0; c < 16; c += 2)
            acc[(16 * h + c) / 2] = add2(
                acc[(16 * h + c) / 2],
                mod_p2(pack2(__uint_as_float(r[h & 1][c]), __uint_as_float(r[h & 1][c + 1])), np2, inv2, mg2, nmg2));
        }
        if (FOLD && --left == 0) {
          left = g.fold;
#pragma unroll
          for (int c = 0; c < TC_CPT / 2; ++c) acc[c] = mod_p2(acc[c], np2, inv2, mg2, nmg2);
        }
      }
      if (!ok) break;
      // (sum mod p) times the modulus' weight, mod p, in [0, p): the term of
      // the Chinese remainder sum
      const f32x2 w2 = pack2(tab.q[t.mod], tab.q[t.mod]);
      unsigned short* R = g.R + (((long long)t.z * g.nmod + t.mod) * g.n) * ldr + t.mt * TC_BM + 32 * lq + lane;
      const int col0 = t.nt * TC_BN + TC_CPT * ch;
#pragma unroll
      for (int c = 0; c < TC_CPT; c += 2) {
        const f32x2 z2 = mod_p2(fma2(mod_p2(acc[c / 2], np2, inv2, mg2, nmg2), w2, 0ull), np2, inv2, mg2, nmg2);
        float v[2];
        unpack2(z2, v[0], v[1]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float x = v[u] < 0.0f ? v[u] + p : v[u];
          // the integer, from the low bits of x + 2^23
          if (col0 + c + u < g.n)
            R[(long long)(col0 + c + u) * ldr] = (unsigned short)(__float_as_uint(x + 8388608.0f) & 0xFFFFu);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---- operands: exponents of rows of op(A) (columns of op(B)) and residues

// Per-term weights w_j of a grouped sum, passed by value (no host-to-device
// copy, so the whole product can be captured in a CUDA graph).
struct TermWeights {
  double w[MAX_SUM];
};

struct ConvArgs {
  int rows, K, op;  // op(X): rows x K
  const double* X;
  int ld, bdiv;
  long long sX, sXj;
  int nrb;                   // 128-row blocks stored
  __nv_bfloat16* out;
  int* e;                    // row exponents, [problem][128 nrb]
  int* part;                 // ... of the k segments, [problem][segment][128 nrb]
  int sgn;                   // sign of the inner-dimension balance exponent
  int unit;                  // all weights are 1
  TermWeights w;
};

constexpr int CV_ROWS = 32;  // rows of a CTA of the conversion

// One side of a product: what the two conversion kernels need of it.
struct ConvSide {
  int op, rows, K, nrb, bsgn;
  bool unit;
  const double* X;        // of this problem
  long long si, sk, sXj;  // strides of i, k and the term
  __device__ ConvSide(const ConvArgs& a, int b, int es)
      : op(a.op), rows(a.rows), K(a.K), nrb(a.nrb), bsgn(a.sgn), unit(a.unit),
        X(a.X + (long long)(b / a.bdiv) * a.sX * es), si(a.op == OP_N ? es : (long long)a.ld * es),
        sk(a.op == OP_N ? (long long)a.ld * es : es), sXj(a.sXj) {}
};

// Largest exponent of every row of op(X) over all terms and one k segment,
// |x| < 2^e for the biased exponent E = e + 1022 (INT_MIN: no normal entry), to
// part[problem][segment][row].  Both operands of a product in one launch
// (blockIdx.y); eight threads share a row.
__global__ void __launch_bounds__(256) tc_exp_kernel(const __grid_constant__ ConvArgs a0,
                                                     const __grid_constant__ ConvArgs a1, int nsum, int segs, int es,
                                                     const int* ek, int ekpad) {
  __shared__ int rmax[CV_ROWS];
  const bool second = blockIdx.y != 0;
  const int b = blockIdx.z, tid = threadIdx.x;
  const ConvSide c(second ? a1 : a0, b, es);
  const int rblk = blockIdx.x / segs, seg = blockIdx.x % segs, i0 = rblk * CV_ROWS;
  if (i0 >= 128 * c.nrb) return;
  const int* ekb = ek ? ek + (long long)b * ekpad : nullptr;
  if (tid < CV_ROWS) rmax[tid] = INT_MIN;
  __syncthreads();
  const int row = c.op == OP_N ? tid % CV_ROWS : tid / 8;
  const int kb = (int)((long long)c.K * seg / segs) + (c.op == OP_N ? tid / CV_ROWS : tid % 8),
            ke = (int)((long long)c.K * (seg + 1) / segs);
  int mx = INT_MIN;
  if (i0 + row < c.rows)
    for (int j = 0; j < nsum; ++j) {
      const double* X = c.X + j * c.sXj + (i0 + row) * c.si;
      const double w = second ? 1.0 : a0.w.w[j];
#pragma unroll 8
      for (int k = kb; k < ke; k += 8) {
        double v = X[k * c.sk];
        if (!c.unit) v *= w;
        const int E = (int)((__double_as_longlong(v) >> 52) & 0x7FF);
        const int bal = ekb ? (ekb[k] > -2000 ? c.bsgn * ekb[k] : 0) : 0;
        mx = max(mx, E > 0 ? E - 1022 + bal : INT_MIN);
      }
    }
  if (mx != INT_MIN) atomicMax(&rmax[row], mx);
  __syncthreads();
  if (tid < CV_ROWS) (second ? a1.part : a0.part)[((long long)b * segs + seg) * 128 * c.nrb + i0 + tid] = rmax[tid];
}

// Residues of 32 rows of op(X) and one k segment, all terms.  Integers and
// residues use integer and FP32 instructions only: the two FP64 scalings and
// the conversion of an entry would cost twice the 14 residues.
__global__ void __launch_bounds__(256, 2) tc_convert_kernel(const __grid_constant__ ConvArgs a0,
                                                            const __grid_constant__ ConvArgs a1, int nsum, int nkb,
                                                            int segs, int esegs, int es, const int* ek, int ekpad,
                                                            const __grid_constant__ RnsTab tab) {
  __shared__ double tile[CV_ROWS][76];  // 8 entries, 1 unused: fewer bank conflicts
  __shared__ int rmax[CV_ROWS];
  const bool second = blockIdx.y != 0;
  const int b = blockIdx.z, tid = threadIdx.x;
  const ConvSide c(second ? a1 : a0, b, es);
  const int op = c.op, rows = c.rows, K = c.K, nrb = c.nrb, bsgn = c.bsgn;
  const bool unit = c.unit;
  const double* const X0 = c.X;
  const long long si = c.si, sk = c.sk, sXj = c.sXj;
  const int rblk = blockIdx.x / segs, seg = blockIdx.x % segs, i0 = rblk * CV_ROWS;
  if (i0 >= 128 * nrb) return;
  const int* ekb = ek ? ek + (long long)b * ekpad : nullptr;
  if (tid < CV_ROWS) {
    const int* part = (second ? a1.part : a0.part) + (long long)b * esegs * 128 * nrb + i0 + tid;
    int mx = INT_MIN;
    for (int q = 0; q < esegs; ++q) mx = max(mx, part[(long long)q * 128 * nrb]);
    rmax[tid] = mx;
    if (seg == 0) (second ? a1.e : a0.e)[(long long)b * 128 * nrb + i0 + tid] = mx == INT_MIN ? 0 : mx;
  }
  __syncthreads();
  // ---- residues: one 16-byte unit (8 consecutive k of a row) per thread and
  // modulus; the next tile is on its way while this one is reduced
  const int r = tid / 8, k8 = tid % 8;
  const int e = rmax[r];
  const int kb0 = (int)((long long)nkb * seg / segs), kb1 = (int)((long long)nkb * (seg + 1) / segs);
  const int per = kb1 - kb0, steps = per * nsum;
  double ahead[8];
  // this thread's entries of a tile: op N: row tid % 32, every 8th k; op T:
  // k tid % 64, every 4th row
  const int fr = op == OP_N ? tid % CV_ROWS : tid / TC_BK, fk = op == OP_N ? tid / CV_ROWS : tid % TC_BK;
  const int dr = op == OP_N ? 0 : 4, dk = op == OP_N ? 8 : 0;
  auto fetch = [&](int j, int kb) {
    const double* X = X0 + j * sXj + (long long)(i0 + fr) * si + (long long)(kb * TC_BK + fk) * sk;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      ahead[u] = (i0 + fr + dr * u < rows && kb * TC_BK + fk + dk * u < K) ? X[u * (dr * si + dk * sk)] : 0.0;
  };
  __nv_bfloat16* const out0 = second ? a1.out : a0.out;
  int j = 0, kb = kb0;
  if (steps > 0) fetch(0, kb0);
  const f32x2 mg2 = pack2(12582912.0f, 12582912.0f), nmg2 = pack2(-12582912.0f, -12582912.0f);
  for (int it = 0; it < steps; ++it) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int kk = fk + dk * u;
      tile[fr + dr * u][kk + kk / 8] = ahead[u];
    }
    __syncthreads();
    const int jn = kb + 1 < kb1 ? j : j + 1, kn = kb + 1 < kb1 ? kb + 1 : kb0;
    if (it + 1 < steps) fetch(jn, kn);
    const double w = second ? 1.0 : a0.w.w[j];
    f32x2 x0[4], x1[4], x2[4], x3[4];  // 14-bit digits of the integers, signed
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      float d[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        double v = tile[r][k8 * 9 + u + h];
        if (!unit) v *= w;
        const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
        int E = (int)((bits >> 52) & 0x7FF);
        unsigned long long mant = (bits & 0xFFFFFFFFFFFFFull) | (E ? 1ull << 52 : 0ull);
        E = E ? E : 1;
        const int k = kb * TC_BK + k8 * 8 + u + h;
        if (ekb && k < K && ekb[k] > -2000) E += bsgn * ekb[k];
        // |x| 2^(bits - e) = mant 2^s = (mant << 4) 2^(s - 4), s - 4 < 0
        int sh = 4 - (E - 1075 + tab.bits - e);
        if (e == INT_MIN || sh > 60) sh = 60;  // below half a unit (mant << 4 < 2^57)
        const unsigned long long mag = ((mant << 4) + (1ull << (sh - 1))) >> sh;
        const unsigned sgn = (unsigned)(bits >> 32) & 0x80000000u;
        const unsigned lo = (unsigned)mag, hi = (unsigned)(mag >> 32);
        // the bits of 2^23 + digit
        const unsigned f0 = (lo & 16383u) | 0x4B000000u, f1 = ((lo >> 14) & 16383u) | 0x4B000000u,
                       f2 = (__funnelshift_r(lo, hi, 28) & 16383u) | 0x4B000000u, f3 = (hi >> 10) | 0x4B000000u;
        d[h][0] = __uint_as_float(__float_as_uint(__uint_as_float(f0) - 8388608.0f) ^ sgn);
        d[h][1] = __uint_as_float(__float_as_uint(__uint_as_float(f1) - 8388608.0f) ^ sgn);
        d[h][2] = __uint_as_float(__float_as_uint(__uint_as_float(f2) - 8388608.0f) ^ sgn);
        d[h][3] = __uint_as_float(__float_as_uint(__uint_as_float(f3) - 8388608.0f) ^ sgn);
      }
      x0[u / 2] = pack2(d[0][0], d[1][0]);
      x1[u / 2] = pack2(d[0][1], d[1][1]);
      x2[u / 2] = pack2(d[0][2], d[1][2]);
      x3[u / 2] = pack2(d[0][3], d[1][3]);
    }
    const int rb = (i0 + r) / 128, rr = (i0 + r) % 128;
    __nv_bfloat16* out = out0 + ((((long long)b * nsum + j) * nrb + rb) * tab.nmod * nkb + kb) * (long long)TC_CHUNK +
                         rr * 64 + (k8 ^ (rr & 7)) * 8;
#pragma unroll 2
    for (int t = 0; t < tab.nmod; ++t) {
      const f32x2 np2 = pack2(-tab.p[t], -tab.p[t]), inv2 = pack2(tab.inv[t], tab.inv[t]),
                  c1 = pack2(tab.c1[t], tab.c1[t]), c2 = pack2(tab.c2[t], tab.c2[t]), c3 = pack2(tab.c3[t], tab.c3[t]);
      __nv_bfloat162 o[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        // |sum| <= 2^14 (1 + 255 + 255 + 255) < 2^24: exact
        const f32x2 sum = fma2(x3[u], c3, fma2(x2[u], c2, fma2(x1[u], c1, x0[u])));
        float va, vb;
        unpack2(mod_p2(sum, np2, inv2, mg2, nmg2), va, vb);
        o[u] = __floats2bfloat162_rn(va, vb);
      }
      *reinterpret_cast<uint4*>(out + (long long)t * nkb * TC_CHUNK) = *reinterpret_cast<uint4*>(o);
    }
    j = jn;
    kb = kn;
  }
}

// exponent e_k with max |x| < 2^e_k over row k of op(X) (rows x K), for the
// inner-dimension balance
__global__ void __launch_bounds__(256) tc_row_exp_kernel(int rows, int K, int op, const double* X, int ld, long long sX,
                                                         int bdiv, int pad, int* e, int es) {
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= rows) return;
  const double* Xb = X + (long long)(b / bdiv) * sX * es;
  int mx = INT_MIN;
  for (int k = lane; k < K; k += 32) {
    const double v = op == OP_N ? Xb[es * (i + (long long)k * ld)] : Xb[es * (k + (long long)i * ld)];
    const int E = (int)((__double_as_longlong(v) >> 52) & 0x7FF);
    if (E > 0) mx = max(mx, E - 1022);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) e[(long long)b * pad + i] = mx;  // INT_MIN: no normal entry
}

struct CombArgs {
  int m, n, ldr, uplo, tiles_m;
  const unsigned short* R;
  const int *ea, *eb;
  int epA, epB, bstrideA, bstrideB;  // exponents per problem; 0 stride: shared
  double alpha, beta;
  const double* Cin; int ldcin, bdivC; long long sCin;
  double* C; int ldc; long long sC;
  int es;
  const int* err;
};

// C = alpha 2^(ea + eb - 2 bits) x + beta Cin, x = P frac(sum_t R_t / p_t) with
// the fraction in [-1/2, 1/2): the sum of R_t round(2^96 / p_t) mod 2^96, good
// to 2^-85 of P.  A block covers 128 rows x 16 columns, four rows per thread;
// WIDE numbers the column blocks in the grid's first dimension, where there are
// too many for the second (with one numbering for both, a division in each
// block, the kernel lost a fifth of its rate).
// Reads and writes 2 nmod + 8 bytes per entry; bound by the integer pipe
// (three 32 x 32 + 64-bit multiply-adds per modulus).
template <bool WIDE>
__global__ void __launch_bounds__(256) tc_combine_kernel(const CombArgs g, const __grid_constant__ RnsTab tab) {
  const int m0 = (WIDE ? blockIdx.y : blockIdx.x) * TC_BM, c0 = (WIDE ? blockIdx.x : blockIdx.y) * 16, z = blockIdx.z;
  if (g.uplo == 1 && m0 > c0 / TC_BN * TC_BN + TC_BN - 1) return;
  const bool failed = *g.err != 0;
  const int row = m0 + 4 * (threadIdx.x & 31);
  if (row >= g.m) return;
  const int4 ea4 = *reinterpret_cast<const int4*>(g.ea + (long long)z * g.bstrideA * g.epA + row);  // padded to 128 rows
  const int e4[4] = {ea4.x, ea4.y, ea4.z, ea4.w};
  const int* eb = g.eb + (long long)z * g.bstrideB * g.epB;
  const bool aunit = g.alpha == 1.0 || g.alpha == -1.0;
  const unsigned long long asgn = (aunit && g.alpha < 0.0) ? 1ull << 63 : 0ull;
  double* C = g.C + (long long)z * g.sC * g.es;
  const double* Cin = (g.Cin && g.beta != 0.0) ? g.Cin + (long long)(z / g.bdivC) * g.sCin * g.es : nullptr;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int col = c0 + (threadIdx.x >> 5) + 8 * q;
    if (col >= g.n) continue;
    const unsigned short* R = g.R + ((long long)z * tab.nmod * g.n + col) * g.ldr + row;
    const long long step = (long long)g.n * g.ldr;
    unsigned long long s0[4] = {0, 0, 0, 0}, s1[4] = {0, 0, 0, 0};
    unsigned s2[4] = {0, 0, 0, 0};  // the rest wraps
#pragma unroll 7
    for (int t = 0; t < tab.nmod; ++t) {
      const ushort4 v = *reinterpret_cast<const ushort4*>(R + t * step);
      const unsigned x[4] = {v.x, v.y, v.z, v.w};
      const unsigned w0 = tab.C0[t], w1 = tab.C1[t], w2 = tab.C2[t];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        s0[u] += (unsigned long long)x[u] * w0;
        s1[u] += (unsigned long long)x[u] * w1;
        s2[u] += x[u] * w2;
      }
    }
    const int ebc = eb[col];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (row + u >= g.m) continue;
      // mod 2^96 (a whole P drops out): a signed 64-bit and a low 32-bit word
      const unsigned long long mid = s1[u] + (s0[u] >> 32);
      const unsigned top32 = s2[u] + (unsigned)(mid >> 32);
      unsigned long long mh = ((unsigned long long)top32 << 32) | (unsigned)mid;
      unsigned ml = (unsigned)s0[u];
      const unsigned long long sgn = mh & (1ull << 63);
      if (sgn) {
        ml = 0u - ml;
        mh = ~mh + (ml == 0u ? 1ull : 0ull);
      }
      double v = 0.0;
      if (mh | ml) {
        // magnitude (mh 2^32 + ml) = top 2^ex, bit 63 of top set
        unsigned long long top;
        int ex;
        if (mh) {
          const int lz = __clzll((long long)mh);
          top = lz ? (mh << lz) | (((unsigned long long)ml << 32) >> (64 - lz)) : mh;
          ex = 32 - lz;
        } else {
          const int lz = __clz((int)ml) + 32;
          top = (unsigned long long)ml << lz;
          ex = -lz;
        }
        // times P / 2^96, truncated to 64 bits
        unsigned long long prod = __umul64hi(top, tab.Pm);
        int pe = ex + tab.Pe + 64 - 96;
        if (!(prod >> 63)) {
          prod <<= 1;
          --pe;
        }
        v = mag_to_double(prod, pe + e4[u] + ebc - 2 * tab.bits, sgn);
      }
      if (aunit) v = __longlong_as_double(__double_as_longlong(v) ^ (long long)asgn);
      else v *= g.alpha;
      if (Cin) v = fma(g.beta, Cin[(row + u + (long long)col * g.ldcin) * g.es], v);
      if (failed) v = NAN;
      C[(row + u + (long long)col * g.ldc) * g.es] = v;
    }
  }
}

int num_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 152;
  }
  return sms;
}

}  // namespace

thread_local TcState t_tc;

bool tc_will_handle(const GemmArgs<double>& g) {
  if (!(t_tc.enabled && t_tc.ar && ((t_tc.sites >> g.site) & 1u) && g.ksplit == 1)) return false;
  if (g.m < 32 || g.n < 32 || g.k < 32 || g.nsum < 1) return false;
  // Below about 12 M multiply-adds the FP64 pipe is done (40 us, spread over
  // all SMs by small tiles) before the conversions and three launches pay.
  const double work = (double)g.m * g.n * g.k * g.batch * g.nsum * (g.uplo ? 0.5 : 1.0) * (g.kflags ? 0.5 : 1.0);
  return work >= 12e6;
}

size_t tc_gemm_bytes(long long m, long long n, long long k, int nsum) {
  const long long mp = (m + 127) / 128 * 128, np = (n + 127) / 128 * 128, kp = (k + 63) / 64 * 64;
  return (size_t)(2 * TC_MAXMOD * ((mp + np) * kp * nsum + mp * n)) + 4 * 33 * (mp + np) + 8192;
}

void tc_gemm(const GemmArgs<double>& g, cudaStream_t st, Arena& ar, int* err) {
  ProfToken tok = prof_begin(st);  // conversions, products and combination
  const int nsum = std::max(g.nsum, 1);
  const int bits = ((t_tc.reduced_sites >> g.site) & 1u) ? t_tc.reduced_bits : 56;
  RnsTab tab = pick_tab(bits, (double)g.k * nsum);
  tab.bits = bits;
  const size_t mk = ar.mark();
  TcArgs t{};
  t.m = g.m; t.n = g.n; t.nsum = nsum; t.batch = g.batch; t.nmod = tab.nmod;
  t.nrbA = t.tiles_m = ceil_div(g.m, TC_BM);
  t.nrbB = ceil_div(g.n, 128);
  t.tiles_n = ceil_div(g.n, TC_BN);
  t.nkb = ceil_div(g.k, TC_BK);
  t.kpad = t.nkb * TC_BK;
  t.kb_flags = g.kflags;
  t.uplo = g.uplo == 1 ? 1 : 0;
  for (int nt = 0; nt < t.tiles_n; ++nt) t.tiles += tile_rows(t.uplo, nt, t.tiles_m);
  // op(A) and op(B)^T the same matrix (a Gram product Y^* Y): one set of
  // residues and exponents serves both operands
  bool unit = true;
  for (int j = 0; j < nsum; ++j) unit = unit && g.w[j] == 1.0;
  const bool same = g.A == g.B && g.lda == g.ldb && g.sA == g.sB && g.sAj == g.sBj && g.bdivA == g.bdivB &&
                    g.m == g.n && ((g.opA != OP_N) == (g.opB == OP_N)) && unit;
  const int nA = g.sA == 0 ? 1 : g.batch, nB = g.sB == 0 ? 1 : g.batch;
  t.bstrideA = g.sA == 0 ? 0 : 1;
  t.bstrideB = g.sB == 0 ? 0 : 1;
  const long long cA = (long long)t.nrbA * tab.nmod * t.nkb * TC_CHUNK, cB = (long long)t.nrbB * tab.nmod * t.nkb * TC_CHUNK;
  __nv_bfloat16* A = ar.get<__nv_bfloat16>((size_t)cA * nsum * nA);
  __nv_bfloat16* B = same ? A : ar.get<__nv_bfloat16>((size_t)cB * nsum * nB);
  const int epA = 128 * t.nrbA, epB = 128 * t.nrbB;
  int* ea = ar.get<int>((size_t)epA * nA);
  int* eb = same ? ea : ar.get<int>((size_t)epB * nB);
  const int ldr = TC_BM * t.tiles_m;
  unsigned short* R = ar.get<unsigned short>((size_t)g.batch * tab.nmod * g.n * ldr);
  t.A = A; t.B = B; t.R = R; t.err = err;
  t.probe_wait = t_tc.probe_wait;
  t.fold = t_tc.flush_every > 0 ? std::min(t_tc.flush_every, TC_FOLD) : TC_FOLD;
  // inner-dimension balance (one term only): e_k bounds row k of op(B);
  // op(A) D and D^-1 op(B) with D = diag(2^e_k) have the same product, and
  // per-row / per-column scaling of the balanced operands is accurate
  // relative to max_k |a_ik| |b_k.| instead of max |a_i.| max |b_.j|
  int* ek = nullptr;
  if (g.kbal && nsum == 1 && !same && nA == g.batch && nB == g.batch) {
    ek = ar.get<int>((size_t)t.kpad * g.batch);
    tc_row_exp_kernel<<<dim3(ceil_div(g.k, 8), g.batch), 256, 0, st>>>(
        g.k, g.n, g.opB == OP_N ? OP_N : OP_T, g.B, g.ldb, g.sB, g.bdivB, t.kpad, ek, g.es);
    ZCSD_LAUNCH();
  }
  // op(A): rows = m, K = k;  op(B)^T: rows = n, K = k  (op(B)^T = B^T for op N, B for op T)
  ConvArgs a{}, b{};
  a.rows = g.m; a.K = g.k; a.op = g.opA == OP_N ? OP_N : OP_T;
  a.X = g.A; a.ld = g.lda; a.bdiv = g.bdivA; a.sX = g.sA; a.sXj = g.sAj;
  a.nrb = t.nrbA; a.out = A; a.e = ea; a.sgn = 1; a.unit = unit;
  b.rows = g.n; b.K = g.k; b.op = g.opB == OP_N ? OP_T : OP_N;
  b.X = g.B; b.ld = g.ldb; b.bdiv = g.bdivB; b.sX = g.sB; b.sXj = g.sBj;
  b.nrb = t.nrbB; b.out = B; b.e = eb; b.sgn = -1; b.unit = 1;
  for (int j = 0; j < MAX_SUM; ++j) {
    a.w.w[j] = g.w[j];
    b.w.w[j] = 1.0;
  }
  // k segments of a row block, about four CTAs per SM (1024^3: 38 us with one
  // kernel for both passes, whose segments repeated the exponent pass)
  const int blocks = 4 * (t.nrbA * nA + (same ? 0 : t.nrbB * nB));
  const int segs = std::max(1, std::min({t.nkb, 32, 4 * num_sms() / blocks}));
  a.part = ar.get<int>((size_t)epA * nA * segs);
  b.part = same ? a.part : ar.get<int>((size_t)epB * nB * segs);
  auto convert = [&](const ConvArgs& x, const ConvArgs& y, int sides, int probs) {
    const int rblk = 4 * std::max(x.nrb, sides == 2 ? y.nrb : 0);
    tc_exp_kernel<<<dim3(rblk * segs, sides, probs), 256, 0, st>>>(x, y, nsum, segs, g.es, ek, t.kpad);
    ZCSD_LAUNCH();
    tc_convert_kernel<<<dim3(rblk * segs, sides, probs), 256, 0, st>>>(x, y, nsum, t.nkb, segs, segs, g.es, ek, t.kpad,
                                                                       tab);
    ZCSD_LAUNCH();
  };
  if (same) {
    convert(a, a, 1, nA);
  } else if (nA == nB) {
    convert(a, b, 2, nA);
  } else {
    convert(a, a, 1, nA);
    convert(b, b, 1, nB);
  }
  static std::once_flag attr_once;
  std::call_once(attr_once, [] {
    cudaFuncSetAttribute(tc_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(tc_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  });
  const long long items = (long long)t.tiles * tab.nmod * g.batch;
  const int grid = (int)std::min<long long>(items, num_sms());
  const bool fold = (long long)t.nkb * nsum > (long long)t.fold * TC_DRAIN;
  if (!fold) tc_gemm_kernel<false><<<grid, TC_THREADS, TC_SMEM, st>>>(t, tab);
  else tc_gemm_kernel<true><<<grid, TC_THREADS, TC_SMEM, st>>>(t, tab);
  ZCSD_LAUNCH();
  CombArgs c{};
  c.m = g.m; c.n = g.n; c.ldr = ldr; c.uplo = t.uplo; c.tiles_m = t.tiles_m;
  c.R = R; c.ea = ea; c.eb = eb; c.epA = epA; c.epB = same ? epA : epB;
  c.bstrideA = t.bstrideA; c.bstrideB = t.bstrideB;
  c.alpha = re(g.alpha); c.beta = re(g.beta);
  c.Cin = g.Cin; c.ldcin = g.ldcin; c.bdivC = g.bdivC; c.sCin = g.sCin;
  c.C = g.C; c.ldc = g.ldc; c.sC = g.sC; c.es = g.es; c.err = err;
  const int cblk = ceil_div(g.n, 16);
  if (cblk <= 65535) tc_combine_kernel<false><<<dim3(t.tiles_m, cblk, g.batch), 256, 0, st>>>(c, tab);
  else tc_combine_kernel<true><<<dim3(cblk, t.tiles_m, g.batch), 256, 0, st>>>(c, tab);
  ZCSD_LAUNCH();
  if (tok.slot >= 0) {
    // FP64-equivalent multiply-add work over the tiles executed
    double fma = 0.0;
    for (int by = 0; by < t.tiles_n; ++by)
      for (int bx = 0; bx < tile_rows(t.uplo, by, t.tiles_m); ++bx) {
        const int m0 = bx * TC_BM, n0 = by * TC_BN;
        int kb = 0, ke = g.k;
        if (g.kflags & K_FROM_COL) kb = std::max(kb, n0);
        if (g.kflags & K_FROM_ROW) kb = std::max(kb, m0);
        if (g.kflags & K_TO_COL) ke = std::min(ke, n0 + TC_BN);
        if (g.kflags & K_TO_ROW) ke = std::min(ke, m0 + TC_BM);
        if (ke > kb) fma += (double)std::min(TC_BM, g.m - m0) * std::min(TC_BN, g.n - n0) * (ke - kb);
      }
    prof_end(tok, st, PK_TC, 2.0 * fma * nsum * g.batch, g.site);
  }
  ar.release(mk);
}

bool tc_will_handle_complex(const GemmArgs<z64>& g) {
  // one complex product = two real grouped sums over the interleaved parts;
  // grouped complex sums and the inner-dimension-balanced product stay on
  // the FP64 pipe, as do complex alpha / beta
  if (g.nsum != 1 || g.kbal || g.alpha.y != 0.0 || g.beta.y != 0.0) return false;
  GemmArgs<double> r;
  r.m = g.m; r.n = g.n; r.k = g.k; r.site = g.site; r.ksplit = std::max(1, g.ksplit);
  r.batch = g.batch; r.uplo = g.uplo; r.kflags = g.kflags;
  r.nsum = 4;  // its work in real multiply-adds
  return tc_will_handle(r);
}

void tc_gemm_complex(const GemmArgs<z64>& g, cudaStream_t st, Arena& ar, int* err) {
  // op(A) = A, A^T or A^*: Re op(A) = op'(Re A), Im op(A) = sA op'(Im A)
  // with op' the real N / T and sA = -1 for the conjugate transpose
  const double sa = g.opA == OP_C ? -1.0 : 1.0, sb = g.opB == OP_C ? -1.0 : 1.0;
  GemmArgs<double> r;
  r.m = g.m; r.n = g.n; r.k = g.k;
  r.opA = g.opA == OP_N ? OP_N : OP_T;
  r.opB = g.opB == OP_N ? OP_N : OP_T;
  r.lda = g.lda; r.sA = g.sA; r.ldb = g.ldb; r.sB = g.sB;
  r.ldcin = g.ldcin; r.sCin = g.sCin; r.ldc = g.ldc; r.sC = g.sC;
  r.batch = g.batch; r.bdivA = g.bdivA; r.bdivB = g.bdivB; r.bdivC = g.bdivC;
  r.uplo = g.uplo; r.kflags = g.kflags; r.site = g.site; r.ksplit = g.ksplit;
  r.alpha = g.alpha.x; r.beta = g.beta.x;
  r.nsum = 2;
  r.es = 2;
  const double* A = reinterpret_cast<const double*>(g.A);
  const double* B = reinterpret_cast<const double*>(g.B);
  const double* Ci = reinterpret_cast<const double*>(g.Cin);
  double* C = reinterpret_cast<double*>(g.C);
  // Re C = Re op(A) Re op(B) - Im op(A) Im op(B)
  GemmArgs<double> re_ = r;
  re_.A = A; re_.sAj = 1;
  re_.B = B; re_.sBj = 1;
  re_.w[0] = 1.0; re_.w[1] = -sa * sb;
  re_.Cin = Ci; re_.C = C;
  tc_gemm(re_, st, ar, err);
  // Im C = Re op(A) Im op(B) + Im op(A) Re op(B)
  GemmArgs<double> im_ = r;
  im_.A = A; im_.sAj = 1;
  im_.B = B + 1; im_.sBj = -1;
  im_.w[0] = sb; im_.w[1] = sa;
  im_.Cin = Ci ? Ci + 1 : nullptr; im_.C = C + 1;
  tc_gemm(im_, st, ar, err);
}

}  // namespace zcsd
