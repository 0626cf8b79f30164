// Tensor-core H psi of a spin sector (real amplitudes): the alpha-hop x beta-hop
// groups of Eq. 2's Jordan-Wigner sum, most of H psi's multiply-adds, as exact
// integer products on the tcgen05 tensor cores.
//
// With amplitudes multiplied by s(Ia, Ib) = (-1)^{pairs of an alpha electron above
// a beta electron}, the element of such a group is a product of one sign per spin
// and a value V[alpha hop, beta hop] (checked group by group on the host). For an
// output alpha string Ia with its source strings Ja(k), k = 0..K-1,
//   T[h, Jb]      = sum_k V[hop k, h] sign_k psi'[Ja(k), Jb]      (a dense product)
//   lambda'[Ia, Jb ^ x_h] += sign(h, Jb) T[h, Jb]                 (h open at Jb)
// where h runs over the undirected beta hops. V splits into the part even under
// the hop's reversal and the odd part; the odd pass runs only where it is not zero.
//
// Single hops' dependence on the other spin's occupations and the mixed part of the
// diagonal join as rows h (an occupied beta qubit) and sources k (an occupied alpha
// qubit). Everything that moves or counts one spin only is a matrix over that spin's
// strings, applied as a dense product (k_tc_onespin_gemm).
//
// What bounds it and why this form: the direct sum (k_hpsi_str) needs one FP64
// multiply-add and about six shared-memory or L1 accesses per (output, group), and
// GB300's FP64 rate is 1.2 TFLOP/s. Cut into 7 balanced digits of 9 bits (62 bits
// below the largest magnitude), both operands are integers of at most 2^8 that fp16
// holds exactly, 28 digit products (levels i + j <= 6) give every bit that matters,
// and a level's FP32 sum is exact: 64 products of 2^16 reach 2^22 and up to four of
// them per level 2^24 (the levels below 2^-36 may round in their last bit). Levels
// are combined in 64-bit integers and lambda is accumulated in a per-row fixed point
// of 62 bits, so no result depends on any order. Measured against the direct sum, H
// psi alone (one GB300): 85.2 -> 15.1 ms at 30 qubits (9.0M states), 25.0 -> 2.9 ms at
// 26 qubits and 11 electrons (2.2M), 7.0 -> 0.93 ms at 24 qubits and 10 electrons. (The
// kernels for one instance only, with their plan by value, took 11.1, 2.6 and 0.72 ms: the
// instance lists of the batch form cost them registers, k_tc_onespin_gemm above all.)
//
// In norm the error against 64-bit sums stays that of the direct kernels. Entry by entry
// it does not follow the entry's size: psi and V are fixed point below their row's largest
// magnitude, so an entry is off by up to 2^-49 of the largest |V| times the largest |psi|
// that its row sums (vectors over 26 decades: 2^-48.8 to 2^-49.7), where a direct sum's
// error shrinks with its terms.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "vqe_internal.h"
#include "vqe_device.cuh"

namespace vqe {
namespace {

constexpr int kDig = kTcDigits;       // digits per operand
constexpr int kTileN = 64;            // beta strings per tile
constexpr int kRows = 128;            // beta hops per tile (TMEM lanes)
constexpr int kChunkK = 64;           // source alpha strings per pass
constexpr int kReadWarps = 16;        // read the sums from TMEM: warp w the lanes of w % 4, columns of w / 4
constexpr int kThreads = 32 * (kReadWarps + 5);  // then four loading warps and one that issues the products
constexpr uint32_t kABytes = kRows * kChunkK * 2;    // one digit of A
constexpr uint32_t kBBytes = kTileN * kChunkK * 2;   // one digit of a B tile
constexpr int kMaxStages = 12;
constexpr int kLag = 3;               // copy groups a loading thread keeps in flight

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Waits for a barrier's phase for at most two seconds; then, or once another wait
// of the block ran out, marks the block dead and returns (its row becomes NaN).
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* dead,
                                          unsigned long long budget_ns = 2000000000ull) {
  if (mbar_try(bar, parity)) return;
  const unsigned long long t0 = now_ns();
  for (int it = 0; it < (1 << 28); ++it) {
    if (mbar_try(bar, parity)) return;
    if ((it & 255) == 255) {
      if (*dead) return;
      if (now_ns() - t0 > budget_ns) break;
    }
  }
  *dead = 1;
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_ld4(uint32_t addr, float* v) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory operand descriptor: 128-byte swizzle, 8-row groups of 1,024 bytes.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  return uint64_t((addr & 0x3FFFFu) >> 4) | (uint64_t(1024 >> 4) << 16) | (uint64_t(1024 >> 4) << 32) |
         (uint64_t(1) << 46) | (uint64_t(2) << 61);
}
// fp16 x fp16 -> FP32, M = 128, N = n, A with K contiguous, B with N (b_n) or K contiguous
__device__ __forceinline__ uint32_t idesc_of(int n, bool b_n = true) {
  return (1u << 4) | (b_n ? 1u << 16 : 0u) | (uint32_t(n >> 3) << 17) | (uint32_t(kRows >> 4) << 24);
}

// One thread of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred P;\n elect.sync _|P, 0xffffffff;\n selp.u32 %0, 1, 0, P;\n}" : "=r"(p));
  return p != 0;
}
// The products of B digit J with A digits 0..6-J over KS steps of 16 sources, each
// into its level's columns. Straight-line code with constant offsets: issuing, not
// the tensor core, bounds a loop that computes its descriptors (120 clocks a product
// against 48).
template <int KS, int J>
__device__ __forceinline__ void issue_digit(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id) {
#pragma unroll
  for (int i = 0; i + J < kDig; ++i)
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
      tc_mma(tmem + uint32_t(i + J) * kTileN, a + uint64_t(i * (kABytes >> 4) + ks * 2), b + uint64_t(ks * 128), id,
             (J > 0 || ks > 0) ? 1u : 0u);
}
template <int J>
__device__ __forceinline__ void issue_digit(int ksteps, uint32_t tmem, uint64_t a, uint64_t b, uint32_t id) {
  switch (ksteps) {
    case 1: issue_digit<1, J>(tmem, a, b, id); break;
    case 2: issue_digit<2, J>(tmem, a, b, id); break;
    case 3: issue_digit<3, J>(tmem, a, b, id); break;
    default: issue_digit<4, J>(tmem, a, b, id); break;
  }
}

// ---------------------------------------------------------------- fixed point
constexpr int kBadExp = 1 << 20;  // a row holding an infinity or a NaN

// smallest e with |v| < 2^e (v finite; zero and subnormals give -1022)
__device__ __forceinline__ int exp_above(double v) {
  return int((__double_as_longlong(v) >> 52) & 0x7ff) - 1022;
}
// round(x * 2^(62 - e)) for |x| < 2^e, in integers (subnormals count as zero)
__device__ __forceinline__ long long to_fix(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int be = int((b >> 52) & 0x7ff);
  if (be == 0) return 0;
  const int sh = e - (be - 1022);
  if (sh > 62) return 0;
  long long m = ((b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll) << 9;  // 2^62 * the significand in [1/2, 1)
  if (sh > 0) m = (m + (1ll << (sh - 1))) >> sh;
  return b < 0 ? -m : m;
}
__device__ __forceinline__ long long shift_round(long long v, int sh) {
  if (sh <= 0) return v;
  if (sh > 62) return 0;
  return (v + (1ll << (sh - 1))) >> sh;
}
// The level sums v[0..6] of one element (weights 2^(-9 l)) in units of 2^-(46 - de)
// of level 0, de = shl + 1 = 28 - shh.
__device__ __forceinline__ long long combine(float v0, float v1, float v2, float v3, float v4, float v5, float v6,
                                             int shh, int shl, long long rnd) {
  const long long hi = (static_cast<long long>(__float2int_rn(v0)) << 18) +
                       (static_cast<long long>(__float2int_rn(v1)) << 9) + __float2int_rn(v2);
  const long long lo = (static_cast<long long>(__float2int_rn(v3)) << 18) +
                       (static_cast<long long>(__float2int_rn(v4)) << 9) + __float2int_rn(fmaf(v6, 0x1p-9f, v5));
  return (hi << shh) + ((lo + rnd) >> shl);
}
// Balanced base-512 digits of v, |v| <= 2^62: v = sum_j d[j] 2^(54 - 9 j), |d| <= 256
__device__ __forceinline__ void digits(long long v, int* d) {
#pragma unroll
  for (int j = kDig - 1; j > 0; --j) {
    const int t = ((int(v) + 256) & 511) - 256;
    d[j] = t;
    v = (v - t) >> 9;
  }
  d[0] = int(v);
}
// two digits as fp16, exactly: 1280 + d has unit spacing, then 1280 is taken off
__device__ __forceinline__ uint32_t half2_of(int lo, int hi) {
  const uint32_t u = (0x6500u + uint32_t(lo)) & 0xFFFFu, w = (0x6500u + uint32_t(hi)) << 16;
  const uint32_t both = u | w;
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&both), __float2half2_rn(1280.0f));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// ---------------------------------------------------------------- instances
// A launch serves one instance (many null) or a batch: instance and work item come
// from the list `work` (tile and row kernels) or from blockIdx.y.
__device__ __forceinline__ TcScratch scratch_of(const TcInst& I, char* ws) {
  TcScratch s;
  s.dig = reinterpret_cast<uint16_t*>(ws + I.off.dig);
  s.one_a = reinterpret_cast<uint16_t*>(ws + I.off.one_a);
  s.one_b = reinterpret_cast<uint16_t*>(ws + I.off.one_b);
  s.pexp = reinterpret_cast<int*>(ws + I.off.pexp);
  s.aexp = reinterpret_cast<int*>(ws + I.off.aexp);
  s.ade = reinterpret_cast<int*>(ws + I.off.ade);
  s.bexp = reinterpret_cast<int*>(ws + I.off.bexp);
  s.bde = reinterpret_cast<int*>(ws + I.off.bde);
  s.vi = reinterpret_cast<long long*>(ws + I.off.vi);
  s.vexp = reinterpret_cast<int*>(ws + I.off.vexp);
  s.vodd = reinterpret_cast<int*>(ws + I.off.vodd);
  s.vsum = reinterpret_cast<double*>(ws + I.off.vsum);
  s.row = reinterpret_cast<int4*>(ws + I.off.row);
  s.lost = reinterpret_cast<int*>(s.row + I.tc.Da);
  return s;
}

// ---------------------------------------------------------------- operand preparation
// Values of one alpha hop against every beta hop: even and odd parts in fixed
// point below the item's largest magnitude, that exponent, and sum |even| + |odd|.
__global__ void __launch_bounds__(256) k_tc_values(const TcInst* __restrict__ many, const TcInst one, char* ws) {
  const TcInst& I = many ? many[blockIdx.y] : one;
  const TcPlan& tc = I.tc;
  if (int(blockIdx.x) >= tc.items) return;
  const TcScratch sc = scratch_of(I, ws);
  const double* vals = I.vals;
  __shared__ double rs[8];
  __shared__ int rm[8];
  const int a = blockIdx.x, R = tc.MT * kRows;
  double sum = 0.0;
  int top = -1022, odd = 0;
  for (int m = threadIdx.x; m < R; m += blockDim.x) {
    const int2 sl = tc.vslot[int64_t(a) * R + m];
    const double v0 = sl.x == -1 ? 0.0 : sflip(vals[sl.x & 0x7fffffff], int(uint32_t(sl.x) >> 31));
    const double v1 = sl.y == -1 ? 0.0 : sflip(vals[sl.y & 0x7fffffff], int(uint32_t(sl.y) >> 31));
    const double ev = 0.5 * (v0 + v1), od = 0.5 * (v0 - v1);
    sum += fabs(ev) + fabs(od);
    top = max(top, max(exp_above(ev), exp_above(od)));
    odd |= od != 0.0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    odd |= __shfl_xor_sync(0xffffffffu, odd, o);
  }
  if ((threadIdx.x & 31) == 0) {
    rs[threadIdx.x >> 5] = sum;
    rm[threadIdx.x >> 5] = top * 2 + (odd ? 1 : 0);
  }
  __syncthreads();
  sum = 0.0;
  top = -1022;
  odd = 0;
  for (int w = 0; w < int(blockDim.x >> 5); ++w) {
    sum += rs[w];
    odd |= rm[w] & 1;
    top = max(top, rm[w] >> 1);
  }
  const bool bad = top > 1023;  // an infinity or a NaN among the values
  for (int m = threadIdx.x; m < R; m += blockDim.x) {
    const int2 sl = tc.vslot[int64_t(a) * R + m];
    const double v0 = sl.x == -1 ? 0.0 : sflip(vals[sl.x & 0x7fffffff], int(uint32_t(sl.x) >> 31));
    const double v1 = sl.y == -1 ? 0.0 : sflip(vals[sl.y & 0x7fffffff], int(uint32_t(sl.y) >> 31));
    sc.vi[int64_t(a) * R + m] = bad ? 0 : to_fix(0.5 * (v0 + v1), top);
    sc.vi[int64_t(tc.items + a) * R + m] = bad ? 0 : to_fix(0.5 * (v0 - v1), top);
  }
  if (threadIdx.x == 0) {
    if (a == 0) *sc.lost = 0;  // the kernels after this one set it
    sc.vexp[a] = bad ? kBadExp : top;
    sc.vodd[a] = odd;
    sc.vsum[a] = sum;
  }
}

// The alpha string's sign mask: beta qubits below an odd number of its electrons.
__device__ __forceinline__ uint32_t sign_mask(uint32_t ka) {
  uint32_t o = 0;
  while (ka) {
    o ^= ((ka & (0u - ka)) - 1u) & 0xAAAAAAAAu;
    ka &= ka - 1u;
  }
  return o;
}

// Digits of one row of psi' (s times psi) below the row's largest magnitude.
// Bound by its writes: 14 bytes per amplitude for 8 read.
__global__ void __launch_bounds__(256) k_tc_digits(const TcInst* __restrict__ many, const TcInst one, char* ws) {
  const TcInst& I = many ? many[blockIdx.y] : one;
  const TcPlan& tc = I.tc;
  if (int(blockIdx.x) >= tc.Da) return;
  const TcScratch sc = scratch_of(I, ws);
  const uint32_t *ka = I.ka, *kb = I.kb;
  const double* psi_am = reinterpret_cast<const double*>(ws + I.off.psi_am);
  __shared__ int rm[8];
  const int ja = blockIdx.x, tid = threadIdx.x;
  const double* row = psi_am + int64_t(ja) * tc.Db;
  int top = -1022;
  for (int j = tid; j < tc.Db; j += blockDim.x) top = max(top, exp_above(row[j]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if ((tid & 31) == 0) rm[tid >> 5] = top;
  __syncthreads();
  top = rm[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) top = max(top, rm[w]);
  const bool bad = top > 1023;
  if (tid == 0) sc.pexp[ja] = bad ? kBadExp : top;
  const uint32_t om = sign_mask(__ldg(ka + ja));
  const int64_t stride = int64_t(tc.Da) * tc.DbP;
  uint16_t* out = sc.dig + int64_t(ja) * tc.DbP;
  for (int j0 = tid * 8; j0 < tc.DbP; j0 += int(blockDim.x) * 8) {
    uint4 w[kDig];
    uint32_t* wp = reinterpret_cast<uint32_t*>(w);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      int d0[kDig], d1[kDig];
      const int j = j0 + 2 * t;
      const long long v0 = (j < tc.Db && !bad) ? neg_if(to_fix(row[j], top), parity32(__ldg(kb + j) & om)) : 0;
      const long long v1 =
          (j + 1 < tc.Db && !bad) ? neg_if(to_fix(row[j + 1], top), parity32(__ldg(kb + j + 1) & om)) : 0;
      digits(v0, d0);
      digits(v1, d1);
#pragma unroll
      for (int s = 0; s < kDig; ++s) wp[s * 4 + t] = half2_of(d0[s], d1[s]);
    }
#pragma unroll
    for (int s = 0; s < kDig; ++s) *reinterpret_cast<uint4*>(out + s * stride + j0) = w[s];
  }
}

// ---------------------------------------------------------------- the product kernel
struct TcShared {          // after the operand buffers and the lambda row
  uint64_t full[kMaxStages], empty[kMaxStages], tfull, tempty, last;
  uint32_t tmem;
  int dead, bad, odd, shift_hi, shift_lo, e;
  uint32_t src[kChunkK];   // source row
  int32_t item[kChunkK];
  int32_t sh[kChunkK];     // shift of the item's values | sign << 16
};

// One output alpha string at a time per block: its 128 x 64 operand A (rows h, sources
// k; 112 KB of digits) stays in shared memory while tiles of 64 beta strings stream
// through a ring of 8 KB stages (one digit each); a tile's seven levels fill 448 of
// the 512 TMEM columns, so reading a tile out does not overlap its successor's
// products. At 30 qubits 7.2 ms: 28 x 4 products of 48 clocks per tile (their shared
// memory reads bound them at N = 64; 64 clocks would do N = 128), then the read-out,
// bound by the 16-per-clock float-to-integer conversions. Sixteen reading warps
// against four: 16.1 -> 7.2 ms, together with products issued from straight-line code. Counters at 24 qubits and 10 electrons (543 us): tensor pipe
// active 19 % of the cycles, issue slots 34 %, DRAM 15 MB; the rest is waiting between the
// two, which share the tensor memory.
__global__ void __launch_bounds__(kThreads, 1)
k_tc_hops(const TcInst* __restrict__ many, const TcInst one, char* ws, const int2* __restrict__ work, int n_work,
          int stages, int lam_len, const TcCtl ctl) {
  extern __shared__ __align__(1024) unsigned char raw[];
  unsigned char* base = raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u);
  unsigned char* sA = base;
  unsigned char* sB = sA + kDig * kABytes;
  uint32_t* lam_lo = reinterpret_cast<uint32_t*>(sB + uint32_t(stages) * kBBytes);
  uint32_t* lam_hi = lam_lo + lam_len;
  TcShared& S = *reinterpret_cast<TcShared*>(lam_hi + lam_len);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == kReadWarps + 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&S.tmem))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < stages; ++i) {
      mbar_init(smem_u32(&S.full[i]), 128);
      mbar_init(smem_u32(&S.empty[i]), 1);
    }
    mbar_init(smem_u32(&S.tfull), 1);
    mbar_init(smem_u32(&S.tempty), 32 * kReadWarps);
    mbar_init(smem_u32(&S.last), 1);
    S.dead = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // rows of a tile past the last source string meet zero digits of A: they must be finite
  for (uint32_t i = tid; i < uint32_t(stages) * kBBytes / 16; i += kThreads)
    reinterpret_cast<uint4*>(sB)[i] = make_uint4(0, 0, 0, 0);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  if (ctl.probe && blockIdx.x == 0) {  // the wait check: a barrier that nothing reaches before the block's end
    if (tid == 0) mbar_wait(smem_u32(&S.last), 0, &S.dead, static_cast<unsigned long long>(ctl.budget_ns));
    __syncthreads();
  }

  // pipeline positions, kept across rows and passes
  int st = 0;
  uint32_t ph = 0;         // loaders: parity of the empty wait ^ 1; issuer: parity of the full wait
  uint32_t tph = 0;        // tile parity (issuer and readers)

  for (int wk = blockIdx.x; wk < n_work; wk += gridDim.x) {
    const TcInst& I = many ? many[__ldg(&work[wk].x)] : one;
    const int ia = many ? __ldg(&work[wk].y) : wk;
    const TcPlan& tc = I.tc;
    const TcScratch sc = scratch_of(I, ws);
    const uint32_t *ka = I.ka, *kb = I.kb;
    double* lam_am = reinterpret_cast<double*>(ws + I.off.lam_am);
    const int R = tc.MT * kRows;  // entries of dst hold eight strings
    const int n_tiles = tc.DbP / kTileN;
    const int4 scales = __ldg(sc.row + ia);
    if (tid == 0) {
      S.e = scales.y;
      S.shift_hi = 28 - scales.z;
      S.shift_lo = scales.z - 1;
      S.bad = scales.w & 1;
      S.odd = scales.w >> 1;
    }
    auto sources = [&](int kc) {  // of one chunk
      if (tid < kChunkK) {
        const int64_t q = int64_t(ia) * tc.KT + kc * kChunkK + tid;
        const uint32_t kj = __ldg(tc.kj + q);
        const int it = __ldg(tc.kit + q);
        const uint32_t r = kj & 0x7fffffffu;
        S.src[tid] = r;
        S.item[tid] = it;
        S.sh[tid] = min(scales.x - __ldg(sc.vexp + it) - __ldg(sc.pexp + r), 63) | int((kj >> 31) << 16);
      }
    };
    sources(0);
    for (int j = tid; j < tc.DbP; j += kThreads) lam_lo[j] = lam_hi[j] = 0u;
    __syncthreads();
    const int passes = S.bad ? 0 : tc.MT * tc.chunks * (S.odd ? 2 : 1);
    for (int ps = 0; ps < passes; ++ps) {
      const int kc = ps % tc.chunks, mt = (ps / tc.chunks) % tc.MT, od = ps / (tc.chunks * tc.MT);
      const int kcnt = min(kChunkK, tc.K - kc * kChunkK);
      const int ksteps = (kcnt + 15) >> 4;
      if (ps > 0) {
        sources(kc);
        __syncthreads();
      }
      // A: digits of V times the sources' scales, [digit][hop][k], 16 bytes (8 k) at a time
      const long long* vi = sc.vi + int64_t(od) * tc.items * R + mt * kRows;
      for (int q = tid; q < kRows * 2 * ksteps; q += kThreads) {
        const int m = q & (kRows - 1), c = q >> 7;
        uint32_t w[kDig][4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          int d[2][kDig];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int k = c * 8 + t * 2 + u;
            long long v = 0;
            if (k < kcnt) {
              const int sh = S.sh[k];
              v = neg_if(shift_round(__ldg(vi + int64_t(S.item[k]) * R + m), sh & 0xffff), sh >> 16);
            }
            digits(v, d[u]);
          }
#pragma unroll
          for (int s = 0; s < kDig; ++s) w[s][t] = half2_of(d[0][s], d[1][s]);
        }
        unsigned char* p = sA + (m >> 3) * 1024 + (m & 7) * 128 + ((c ^ (m & 7)) << 4);
#pragma unroll
        for (int s = 0; s < kDig; ++s)
          *reinterpret_cast<uint4*>(p + s * kABytes) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
      }
      fence_async();
      __syncthreads();

      if (warp >= kReadWarps && warp < kReadWarps + 4) {
        // loaders: one digit of a tile per stage, rows psi'[Ja(k), 64 columns] with N contiguous
        const int pt = tid - 32 * kReadWarps;
        const int64_t stride = int64_t(tc.Da) * tc.DbP;
        int lag_st = st, pending = 0;
        // hands over every copy in flight (before a wait, which the handed-over stages may end)
        auto flush = [&] {
          cp_wait<0>();
          fence_async();
          for (; pending > 0; --pending) {
            mbar_arrive(smem_u32(&S.full[lag_st]));
            if (++lag_st == stages) lag_st = 0;
          }
        };
        for (int t = 0; t < n_tiles; ++t) {
          for (int j = 0; j < kDig; ++j) {
            if (!mbar_try(smem_u32(&S.empty[st]), ph ^ 1)) {
              flush();
              mbar_wait(smem_u32(&S.empty[st]), ph ^ 1, &S.dead);
            }
            const uint32_t dst = smem_u32(sB) + uint32_t(st) * kBBytes;
            const uint16_t* src = sc.dig + j * stride + t * kTileN;
            for (int q = pt; q < kcnt * 8; q += 128) {
              const int k = q >> 3, c = q & 7;
              cp_async16(dst + uint32_t((k >> 3) * 1024 + (k & 7) * 128 + ((c ^ (k & 7)) << 4)),
                         src + int64_t(S.src[k]) * tc.DbP + c * 8);
            }
            cp_commit();
            if (++pending > kLag) {
              cp_wait<kLag>();
              fence_async();
              mbar_arrive(smem_u32(&S.full[lag_st]));
              if (++lag_st == stages) lag_st = 0;
              --pending;
            }
            if (++st == stages) {
              st = 0;
              ph ^= 1;
            }
          }
        }
        flush();
      } else if (warp == kReadWarps + 4) {
        const uint64_t ad = sdesc(smem_u32(sA)), b0 = sdesc(smem_u32(sB));
        for (int t = 0; t < n_tiles; ++t) {
          mbar_wait(smem_u32(&S.tempty), tph ^ 1, &S.dead);
          const uint32_t id = idesc_of(min(kTileN, (tc.Db - t * kTileN + 15) & ~15));
#pragma unroll
          for (int j = 0; j < kDig; ++j) {
            mbar_wait(smem_u32(&S.full[st]), ph, &S.dead);
            tc_fence_after();
            if (elect_one()) {
              const uint64_t bd = b0 + uint64_t(st) * (kBBytes >> 4);
              switch (j) {
                case 0: issue_digit<0>(ksteps, tmem, ad, bd, id); break;
                case 1: issue_digit<1>(ksteps, tmem, ad, bd, id); break;
                case 2: issue_digit<2>(ksteps, tmem, ad, bd, id); break;
                case 3: issue_digit<3>(ksteps, tmem, ad, bd, id); break;
                case 4: issue_digit<4>(ksteps, tmem, ad, bd, id); break;
                case 5: issue_digit<5>(ksteps, tmem, ad, bd, id); break;
                default: issue_digit<6>(ksteps, tmem, ad, bd, id); break;
              }
              tc_commit(smem_u32(&S.empty[st]));
              if (j == kDig - 1) tc_commit(smem_u32(&S.tfull));
            }
            __syncwarp();
            if (++st == stages) {
              st = 0;
              ph ^= 1;
            }
          }
          tph ^= 1;
        }
      } else {
        // readers: lane = row h; combine the levels and add each open (h, Jb) to lambda'
        constexpr int kCols = kTileN * 4 / kReadWarps;
        const int row = (warp & 3) * 32 + lane, col0 = (warp >> 2) * kCols;
        const uint4* dst = tc.dst + mt * kRows + row;
        const uint32_t taddr = tmem + (uint32_t(warp & 3) << 21) + uint32_t(col0);
        const int shh = S.shift_hi, shl = S.shift_lo;
        const long long rnd = shl > 0 ? (1ll << (shl - 1)) : 0ll;
        for (int t = 0; t < n_tiles; ++t) {
          uint4 ent[kCols / 8];
#pragma unroll
          for (int c = 0; c < kCols / 8; ++c) ent[c] = __ldg(dst + int64_t(t * (kTileN / 8) + col0 / 8 + c) * R);
          mbar_wait(smem_u32(&S.tfull), tph, &S.dead);
          tph ^= 1;
          tc_fence_after();
#pragma unroll
          for (int c0 = 0; c0 < kCols; c0 += 4) {
            float v[kDig][4];
#pragma unroll
            for (int l = 0; l < kDig; ++l) tc_ld4(taddr + uint32_t(l * kTileN + c0), v[l]);
            tc_wait_ld();
            const uint4 e8 = ent[c0 / 8];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint32_t pair = (c0 & 4) ? (c < 2 ? e8.z : e8.w) : (c < 2 ? e8.x : e8.y);
              const uint32_t en = (c & 1) ? pair >> 16 : pair & 0xffffu;
              long long x = combine(v[0][c], v[1][c], v[2][c], v[3][c], v[4][c], v[5][c], v[6][c], shh, shl, rnd);
              if (en >> 15) {
                x = neg_if(x, int((en >> 13) ^ (od ? en >> 14 : 0u)) & 1);
                const uint32_t ib = en & 0x1FFFu, xl = uint32_t(x);
                const uint32_t old = atomicAdd(lam_lo + ib, xl);
                atomicAdd(lam_hi + ib, uint32_t(uint64_t(x) >> 32) + (old + xl < xl ? 1u : 0u));
              }
            }
          }
          tc_fence_before();
          mbar_arrive(smem_u32(&S.tempty));
        }
      }
      __syncthreads();  // every product of the pass has been read
    }
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const bool lost = S.bad || S.dead;
    const int e = S.e - 62;
    const uint32_t om = sign_mask(__ldg(ka + ia));
    for (int j = tid; j < tc.Db; j += kThreads) {
      const long long x = static_cast<long long>((uint64_t(lam_hi[j]) << 32) | lam_lo[j]);
      const int64_t o = int64_t(ia) * tc.Db + j;
      lam_am[o] += lost ? nan : ldexp(sflip(__ll2double_rn(x), parity32(__ldg(kb + j) & om)), e);
    }
    __syncthreads();
  }
  if (warp == kReadWarps + 4) {
    if (lane == 0) {  // nothing of this block is in flight when its tensor memory is given back
      tc_commit(smem_u32(&S.last));
      mbar_wait(smem_u32(&S.last), 0, &S.dead);
      if (S.dead && ctl.status) atomicCAS(ctl.status, 0, ctl.code);
    }
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// ---------------------------------------------------------------- one-spin part
// Scales of output row ia of the product kernel, by one warp: 2^ea above every |V psi'|
// element, 2^e = 2^(ea + de) above every partial sum of lambda'. (Here, beside the row of
// the alpha matrix, four loads' latency passes for all rows at once; in the product kernel
// it passed row by row: H psi of 26 qubits and 11 electrons 2.93 -> 2.87 ms, 24 qubits energy
// and gradient 1.90 -> 1.87 ms.)
__device__ __forceinline__ int4 row_scales(const TcPlan& tc, const TcScratch& sc, int ia, int lane) {
  int top = -100000, bad = 0, odd = 0;
  for (int k = lane; k < tc.K; k += 32) {
    const uint32_t kj = __ldg(tc.kj + int64_t(ia) * tc.KT + k);
    const int it = __ldg(tc.kit + int64_t(ia) * tc.KT + k);
    const int ve = __ldg(sc.vexp + it), pe = __ldg(sc.pexp + (kj & 0x7fffffffu));
    bad |= ve == kBadExp || pe == kBadExp;
    odd |= __ldg(sc.vodd + it);
    top = max(top, ve + pe);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    odd |= __shfl_xor_sync(0xffffffffu, odd, o);
  }
  double sum = 0.0;
  if (!bad)
    for (int k = lane; k < tc.K; k += 32) {
      const uint32_t kj = __ldg(tc.kj + int64_t(ia) * tc.KT + k);
      const int it = __ldg(tc.kit + int64_t(ia) * tc.KT + k);
      const int d = __ldg(sc.vexp + it) + __ldg(sc.pexp + (kj & 0x7fffffffu)) - top;  // <= 0
      // vsum <= 2 R 2^vexp: its mantissa against the item's own scale
      if (d > -200) sum += ldexp(__ldg(sc.vsum + it), d - __ldg(sc.vexp + it));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const int de = max(1, exp_above(sum * 1.0000001));
  return make_int4(top, top + de, de, bad | odd << 1);
}

// Digits of one row of a one-spin matrix (H's terms that move electrons of one
// spin only, and that spin's diagonal): row r as a dense vector of n values, each
// the sum of its table slots, times 2^fold[col] (the source rows' exponents; null:
// 1), below the row's largest magnitude 2^oexp; ode: 2^(oexp + ode) bounds the sum
// of magnitudes. Bound by its writes, 14 bytes per matrix element.
__global__ void __launch_bounds__(256) k_tc_onespin(const TcInst* __restrict__ many, const TcInst one, char* ws,
                                                    int beta) {
  const TcInst& I = many ? many[blockIdx.y] : one;
  const TcOneSpin& os = beta ? I.tc.beta : I.tc.alpha;
  if (int(blockIdx.x) >= os.n) return;
  const TcScratch sc = scratch_of(I, ws);
  const double* vals = I.vals;
  const int* fold = beta ? nullptr : sc.pexp;
  uint16_t* dig = beta ? sc.one_b : sc.one_a;
  int *oexp = beta ? sc.bexp : sc.aexp, *ode = beta ? sc.bde : sc.ade;
  const int ld = beta ? I.tc.DbP : I.tc.DaP;
  extern __shared__ __align__(16) double srow[];
  __shared__ double rs[8];
  __shared__ int rm[8];
  const int r = blockIdx.x, tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  for (int j = tid; j < ld; j += blockDim.x) srow[j] = 0.0;
  __syncthreads();
  if (!beta && w == 7) {
    const int4 scales = row_scales(I.tc, sc, r, lane);
    if (lane == 0) {
      sc.row[r] = scales;
      if ((scales.w & 1) || sc.pexp[r] == kBadExp) *sc.lost = 1;
    }
  }
  const int e0 = __ldg(os.off + r), e1 = __ldg(os.off + r + 1);
  int top = -100000;
  for (int e = e0 + tid; e < e1; e += blockDim.x) {
    const int s0 = __ldg(os.soff + e), s1 = __ldg(os.soff + e + 1);
    double v = 0.0;
    for (int q = s0; q < s1; ++q) {
      const uint32_t sl = __ldg(os.slot + q);
      v += sflip(__ldg(vals + (sl & 0x7fffffffu)), int(sl >> 31));
    }
    const int c = __ldg(os.col + e);
    srow[c] = v;
    const int fe = fold ? __ldg(fold + c) : 0;
    top = max(top, exp_above(v) > 1023 || fe == kBadExp ? kBadExp : exp_above(v) + fe);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (lane == 0) rm[w] = top;
  __syncthreads();
  top = rm[0];
#pragma unroll
  for (int i = 1; i < 8; ++i) top = max(top, rm[i]);
  const bool bad = top == kBadExp;
  double sum = 0.0;
  const int64_t stride = int64_t(os.n) * ld;
  for (int j0 = tid * 8; j0 < ld; j0 += int(blockDim.x) * 8) {
    uint32_t wd[kDig][4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      int d[2][kDig];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int j = j0 + 2 * t + u;
        const double v = srow[j];
        long long x = 0;
        if (v != 0.0 && !bad) {
          const int fe = fold ? __ldg(fold + j) : 0;
          x = to_fix(v, top - fe);
          sum += fabs(static_cast<float>(x)) * 0x1p-62f;
        }
        digits(x, d[u]);
      }
#pragma unroll
      for (int s = 0; s < kDig; ++s) wd[s][t] = half2_of(d[0][s], d[1][s]);
    }
#pragma unroll
    for (int s = 0; s < kDig; ++s)
      *reinterpret_cast<uint4*>(dig + s * stride + int64_t(r) * ld + j0) =
          make_uint4(wd[s][0], wd[s][1], wd[s][2], wd[s][3]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) rs[w] = sum;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < 8; ++i) sum += rs[i];
    if (bad) *sc.lost = 1;
    oexp[r] = top;
    ode[r] = max(1, exp_above(sum * 1.0001));
  }
}

// lambda'[Ia, Ib] (+)= sum_Ja Ha[Ia, Ja] psi'[Ja, Ib] + sum_Jb psi'[Ia, Jb] Hb[Ib, Jb]:
// two dense products over digit matrices, a 128 x 64 tile per block, 64 sources per
// chunk. The direct sums cost one FP64 multiply-add per connected pair (1,003 per
// amplitude at 30 qubits, 15 ms at the FP64 peak). A chunk's seven digit pairs
// (A_s, B_s: 24 KB each) stream through a ring of nine slots in the order 0, 6, 1,
// 5, 2, 4, 3, in which the products i + j <= 6 free them, so most of the next chunk
// is loaded while this one is multiplied and read out.
constexpr int kGemmThreads = 416;  // warps 0-7 read TMEM, 8-11 load, 12 issues the products
constexpr uint32_t kPairBytes = kABytes + kBBytes;
constexpr int kRing = 9;
__device__ __forceinline__ int load_order(int i) { return (0x3425160 >> (4 * i)) & 15; }  // 0 6 1 5 2 4 3

struct GemmShared {
  uint64_t full[kRing], empty[kRing], tfull, tempty, last;
  uint32_t tmem;
  int dead;
  int cexp[kTileN], cde[kTileN];
};

__global__ void __launch_bounds__(kGemmThreads, 1)
k_tc_onespin_gemm(const TcInst* __restrict__ many, const TcInst one, char* ws, const int2* __restrict__ work,
                  int n_work, int add, const TcCtl ctl) {
  extern __shared__ __align__(1024) unsigned char raw[];
  unsigned char* ring = raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u);
  GemmShared& S = *reinterpret_cast<GemmShared*>(ring + kRing * kPairBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 12) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&S.tmem))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) {
      mbar_init(smem_u32(&S.full[i]), 128);
      mbar_init(smem_u32(&S.empty[i]), 1);
    }
    mbar_init(smem_u32(&S.tfull), 1);
    mbar_init(smem_u32(&S.tempty), 256);
    mbar_init(smem_u32(&S.last), 1);
    S.dead = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  int st = 0;
  uint32_t ph = 0, tph = 0;
  for (int wk = blockIdx.x; wk < n_work; wk += gridDim.x) {
    const TcInst& I = many ? many[__ldg(&work[wk].x)] : one;
    const int tile = many ? __ldg(&work[wk].y) : wk;
    const TcPlan& tc = I.tc;
    const TcScratch sc = scratch_of(I, ws);
    const uint32_t *ka = I.ka, *kb = I.kb;
    double* lam_am = reinterpret_cast<double*>(ws + I.off.lam_am);
    const int mts = (tc.Da + kRows - 1) / kRows;
    const int ch0 = tc.DaP / kChunkK, ch1 = tc.DbP / kChunkK;
    const int m0 = (tile % mts) * kRows, n0 = (tile / mts) * kTileN;
    if (warp >= 8 && warp < 12) {
      const int pt = tid - 256;
      int lag_st = st, pending = 0;
      // hands over every copy in flight (before a wait, which the handed-over stages may end)
      auto flush = [&] {
        cp_wait<0>();
        fence_async();
        for (; pending > 0; --pending) {
          mbar_arrive(smem_u32(&S.full[lag_st]));
          if (++lag_st == kRing) lag_st = 0;
        }
      };
      for (int ch = 0; ch < ch0 + ch1; ++ch) {
        const bool part0 = ch < ch0;
        const int k0 = (part0 ? ch : ch - ch0) * kChunkK;
        const uint16_t* ab = part0 ? sc.one_a + k0 : sc.dig + k0;
        const int64_t lda = part0 ? tc.DaP : tc.DbP, sa = int64_t(tc.Da) * lda;
        const uint16_t* bb = part0 ? sc.dig + n0 : sc.one_b + k0;
        const int64_t sb = part0 ? int64_t(tc.Da) * tc.DbP : int64_t(tc.Db) * tc.DbP;
        const int br0 = part0 ? k0 : n0, brl = (part0 ? tc.Da : tc.Db) - 1;
        for (int i = 0; i < kDig; ++i) {
          const int s = load_order(i);
          if (!mbar_try(smem_u32(&S.empty[st]), ph ^ 1)) {
            flush();
            mbar_wait(smem_u32(&S.empty[st]), ph ^ 1, &S.dead);
          }
          const uint32_t dst = smem_u32(ring) + uint32_t(st) * kPairBytes;
#pragma unroll
          for (int u = 0; u < kRows * 8 / 128; ++u) {
            const int q = pt + 128 * u, r = q >> 3, c = q & 7;
            cp_async16(dst + uint32_t(r * 128 + ((c ^ (r & 7)) << 4)),
                       ab + s * sa + int64_t(min(m0 + r, tc.Da - 1)) * lda + c * 8);
          }
#pragma unroll
          for (int u = 0; u < kTileN * 8 / 128; ++u) {
            const int q = pt + 128 * u, r = q >> 3, c = q & 7;
            cp_async16(dst + kABytes + uint32_t(r * 128 + ((c ^ (r & 7)) << 4)),
                       bb + s * sb + int64_t(min(br0 + r, brl)) * tc.DbP + c * 8);
          }
          cp_commit();
          if (++pending > kLag) {
            cp_wait<kLag>();
            fence_async();
            mbar_arrive(smem_u32(&S.full[lag_st]));
            if (++lag_st == kRing) lag_st = 0;
            --pending;
          }
          if (++st == kRing) {
            st = 0;
            ph ^= 1;
          }
        }
      }
      flush();
    } else if (warp == 12) {
      for (int ch = 0; ch < ch0 + ch1; ++ch) {
        const bool part0 = ch < ch0;
        const uint32_t id = idesc_of(kTileN, part0);
        const uint64_t kb_step = part0 ? 128 : 2;
        mbar_wait(smem_u32(&S.tempty), tph ^ 1, &S.dead);
        uint64_t ad[kDig], bd[kDig];
        uint32_t pos[kDig];
        auto mul = [&](int i, int j, bool first) {
#pragma unroll
          for (int ks = 0; ks < kChunkK / 16; ++ks)
            tc_mma(tmem + uint32_t(i + j) * kTileN, ad[i] + uint64_t(ks * 2), bd[j] + ks * kb_step, id,
                   (!first || ks > 0) ? 1u : 0u);
        };
#pragma unroll
        for (int i = 0; i < kDig; ++i) {
          constexpr int order[kDig] = {0, 6, 1, 5, 2, 4, 3};
          const int s = order[i];
          mbar_wait(smem_u32(&S.full[st]), ph, &S.dead);
          tc_fence_after();
          pos[s] = uint32_t(st);
          ad[s] = sdesc(smem_u32(ring)) + uint64_t(st) * (kPairBytes >> 4);
          bd[s] = ad[s] + (kABytes >> 4);
          if (++st == kRing) {
            st = 0;
            ph ^= 1;
          }
          if (elect_one()) {
            mul(0, s, true);
            if (s) mul(s, 0, false);
          }
          __syncwarp();
        }
        if (elect_one()) {
          tc_commit(smem_u32(&S.empty[pos[0]]));
          tc_commit(smem_u32(&S.empty[pos[6]]));
#pragma unroll
          for (int s = 1; s <= 5; ++s) {
            mul(1, s, false);
            if (s > 1) mul(s, 1, false);
          }
          tc_commit(smem_u32(&S.empty[pos[1]]));
          tc_commit(smem_u32(&S.empty[pos[5]]));
#pragma unroll
          for (int s = 2; s <= 4; ++s) {
            mul(2, s, false);
            if (s > 2) mul(s, 2, false);
          }
          tc_commit(smem_u32(&S.empty[pos[2]]));
          tc_commit(smem_u32(&S.empty[pos[4]]));
          mul(3, 3, false);
          tc_commit(smem_u32(&S.empty[pos[3]]));
          tc_commit(smem_u32(&S.tfull));
        }
        __syncwarp();
        tph ^= 1;
      }
    } else {
      const int row = min(m0 + (warp & 3) * 32 + lane, tc.Da - 1);
      const bool live = m0 + (warp & 3) * 32 + lane < tc.Da;
      const int col0 = (warp >> 2) * 32;
      const uint32_t taddr = tmem + (uint32_t(warp & 3) << 21) + uint32_t(col0);
      if (warp >= 6) {  // column scales of the second product
        const int c = tid - 192, ib = min(n0 + c, tc.Db - 1);
        S.cexp[c] = __ldg(sc.bexp + ib);
        S.cde[c] = __ldg(sc.bde + ib);
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const int rexp = __ldg(sc.aexp + row), rde = __ldg(sc.ade + row), pexp = __ldg(sc.pexp + row);
      const uint32_t om = sign_mask(__ldg(ka + row));
      double* out = lam_am + int64_t(row) * tc.Db + n0 + col0;
      for (int part = 0; part < 2; ++part) {
        long long acc[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[c] = 0;
        for (int ch = 0; ch < (part ? ch1 : ch0); ++ch) {
          mbar_wait(smem_u32(&S.tfull), tph, &S.dead);
          tph ^= 1;
          tc_fence_after();
#pragma unroll
          for (int c0 = 0; c0 < 32; c0 += 4) {
            float v[kDig][4];
#pragma unroll
            for (int l = 0; l < kDig; ++l) tc_ld4(taddr + uint32_t(l * kTileN + c0), v[l]);
            tc_wait_ld();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int de = part ? S.cde[col0 + c0 + c] : rde;
              const long long rnd = de > 1 ? 1ll << (de - 2) : 0ll;
              acc[c0 + c] += combine(v[0][c], v[1][c], v[2][c], v[3][c], v[4][c], v[5][c], v[6][c], 28 - de, de - 1, rnd);
            }
          }
          tc_fence_before();
          mbar_arrive(smem_u32(&S.tempty));
        }
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          if (!live || n0 + col0 + c >= tc.Db) continue;
          const int ce = S.cexp[col0 + c];
          const bool lost = S.dead || (part ? ce == kBadExp || pexp == kBadExp : rexp == kBadExp);
          const int e = part ? pexp + ce + S.cde[col0 + c] : rexp + rde;
          const int sg = parity32(__ldg(kb + n0 + col0 + c) & om);
          const double x = lost ? nan : ldexp(sflip(__ll2double_rn(acc[c]), sg), e - 62);
          out[c] = (part || add) ? out[c] + x : x;
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");  // the column scales are read
    }
  }
  __syncthreads();
  if (warp == 12) {
    if (lane == 0) {
      tc_commit(smem_u32(&S.last));
      mbar_wait(smem_u32(&S.last), 0, &S.dead);
      if (S.dead && ctl.status) atomicCAS(ctl.status, 0, ctl.code);
    }
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}
size_t gemm_smem() { return 1024 + size_t(kRing) * kPairBytes + sizeof(GemmShared); }

size_t hops_smem(int DbP, int stages) {
  return 1024 + size_t(kDig) * kABytes + size_t(stages) * kBBytes + size_t(DbP) * 8 + sizeof(TcShared);
}
}  // namespace

// Stages of the loaders' ring that fit next to the operands and the lambda row (0: too few).
int tc_stages(int DbP, size_t smem_limit) {
  int s = kMaxStages;
  while (s > 0 && hops_smem(DbP, s) > smem_limit) --s;
  return s > kLag + 1 ? s : 0;
}

cudaError_t tc_set_smem_limit(size_t bytes) {
  if (bytes < gemm_smem()) return cudaErrorInvalidValue;
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_tc_hops, a, int(bytes));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_tc_onespin_gemm, a, int(bytes));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_tc_onespin, a, int(bytes) - 2048);  // beside its static arrays
  return e;
}

int tc_tiles(const TcPlan& tc) { return (tc.Da + kRows - 1) / kRows * (tc.DbP / kTileN); }

cudaError_t tc_hpsi(const TcBatch& B, const TcInst* one, char* ws, bool add, const TcCtl& ctl, cudaStream_t stream) {
  const TcInst none{};
  const TcInst& o = one ? *one : none;
  const TcInst* many = one ? nullptr : B.insts;
  const unsigned n = one ? 1u : unsigned(B.n);
  k_tc_values<<<dim3(unsigned(B.items), n), 256, 0, stream>>>(many, o, ws);
  k_tc_digits<<<dim3(unsigned(B.Da), n), 256, 0, stream>>>(many, o, ws);
  k_tc_onespin<<<dim3(unsigned(B.Da), n), 256, size_t(B.DaP) * 8, stream>>>(many, o, ws, 0);
  k_tc_onespin<<<dim3(unsigned(B.Db), n), 256, size_t(B.DbP) * 8, stream>>>(many, o, ws, 1);
  const int tg = B.n_tiles < B.sms ? B.n_tiles : B.sms, rg = B.n_rows < B.sms ? B.n_rows : B.sms;
  k_tc_onespin_gemm<<<tg, kGemmThreads, gemm_smem(), stream>>>(many, o, ws, B.tiles, B.n_tiles, add ? 1 : 0, ctl);
  k_tc_hops<<<rg, kThreads, hops_smem(B.DbP, B.stages), stream>>>(many, o, ws, B.rows, B.n_rows, B.stages, B.DbP,
                                                                 ctl);
  return cudaGetLastError();
}

}  // namespace vqe
