// H psi of a large electron-number sector whose Hamiltonian only counts and hops
// (pUCCD's hard-core boson form, Sec. 2.1.2): lambda = (diagonal + sum_{p<q} K_pq hop_pq) psi.
//
// The hops are split into a few passes, each over the hops within a set S of qubits: the
// sector falls into blocks of equal occupation of the other qubits, and a block's
// amplitudes (at most kHopStates) are read into shared memory once per pass. Blocks with
// the same electron count on S share one list of (source, hop) entries per state, which
// stays in L2. The diagonal is a sum of table values of the state's two halves.
//
// What bounds it and why this form: by connectivity rows (k_hpsi) an entry costs a group
// record, a table value, two rank lookups and a scattered read of psi from L2; 24 orbitals
// and 12 pairs (2.7 million states, 145 entries each) took 4.1 ms against 0.65 ms of FP64
// multiply-adds. Here it costs one coalesced 4-byte read, two shared-memory reads and the
// multiply-add: 4.15 -> 1.08 ms, bound by the FP64 pipe and the shared-memory reads.
// (Padding entries are skipped: a state that is not finite must not reach outputs that no
// hop connects it to. Multiplied by 0 instead, they made it 1.30 ms.)
#include <cuda_runtime.h>

#include "vqe_internal.h"
#include "vqe_device.cuh"

namespace vqe {
namespace {

constexpr int kThreads = 512;
constexpr int kAhead = 8;

__device__ __forceinline__ void copy8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Diagonal tables: row 0 by the low half v, row 1 by the high half h (with the constant),
// row 2 + p the part that qubit p of the high half shares with v.
__global__ void __launch_bounds__(256) k_hop_tables(HopDiag g, int n, int lo_bits, const double* __restrict__ vals,
                                                    double* __restrict__ tab) {
  const uint32_t size = 1u << lo_bits, v = blockIdx.x * 256u + threadIdx.x;
  const int row = blockIdx.y;
  if (v >= size) return;
  const double* one = vals + g.slot + 1;
  const double* two = one + g.stride;
  double s = 0.0;
  if (g.slot >= 0) {
    if (row < 2) {
      const int shift = row ? lo_bits : 0;
      if (row == 1) {
        if (v >= (1u << (n - lo_bits))) return;
        s = vals[g.slot];
      }
      for (uint32_t a = (v << shift) & g.counted; a; a &= a - 1) {
        const int p = __ffs(a) - 1;
        s += one[p];
        for (uint32_t b = a & (a - 1); b; b &= b - 1) s += two[p * g.stride + __ffs(b) - 1];
      }
    } else {
      const int p = lo_bits + row - 2;
      if ((g.counted >> p) & 1u)
        for (uint32_t a = v & g.counted; a; a &= a - 1) s += two[(__ffs(a) - 1) * g.stride + p];
    }
  }
  tab[(size_t(row) << lo_bits) + v] = s;
}

// lambda = diagonal psi (0 without a diagonal, also where psi is not finite). Consecutive
// states mostly share the high half.
__global__ void __launch_bounds__(256) k_hop_diag(const uint32_t* __restrict__ sector, int64_t D, int lo_bits,
                                                  int any, const double* __restrict__ tab,
                                                  const double* __restrict__ psi, double* __restrict__ lam) {
  const uint32_t lo_mask = (1u << lo_bits) - 1u;
  for (int64_t r = blockIdx.x * int64_t(256) + threadIdx.x; r < D; r += int64_t(gridDim.x) * 256) {
    const uint32_t k = __ldg(sector + r), h = k >> lo_bits, v = k & lo_mask;
    double s = tab[v] + tab[(size_t(1) << lo_bits) + h];
    for (uint32_t a = h; a; a &= a - 1) s += tab[(size_t(1 + __ffs(a)) << lo_bits) + v];
    lam[r] = any ? s * psi[r] : 0.0;
  }
}

// One pass on one CTA's blocks: lambda += hops of psi.
__global__ void __launch_bounds__(kThreads, 2)
k_hop_blocks(const HopTables T, const HopStep s, const uint32_t* __restrict__ rank_hi,
             const uint32_t* __restrict__ rank_lo, int lo_bits, const double* __restrict__ vals,
             const double* __restrict__ psi, double* __restrict__ lam) {
  extern __shared__ __align__(16) double st[];
  double* hop = st + s.most;
  const uint32_t pad = uint32_t(s.slots) << 16;  // entries from here on are no hops
  const int tid = threadIdx.x;
  const GroupWork w = T.work[s.work0 + blockIdx.x];
  const HopClass c = T.classes[w.cls];
  const int total = c.n * w.count;
  const uint32_t st_a = uint32_t(__cvta_generic_to_shared(st)), lo_mask = (1u << lo_bits) - 1u;
  auto rank_of = [&](int i, int& j) {
    j = c.n == total ? 0 : int(__umulhi(uint32_t(i), c.inv));
    const uint32_t k = __ldg(T.patterns + w.first + j) | __ldg(T.states + c.state0 + i - j * c.n);
    return __ldg(rank_hi + (k >> lo_bits)) + __ldg(rank_lo + (k & lo_mask));
  };
  int j;
#pragma unroll 4
  for (int i = tid; i < total; i += kThreads) copy8(st_a + uint32_t(i) * 8u, psi + rank_of(i, j));
  for (int i = tid; i < s.slots; i += kThreads) hop[i] = vals[__ldg(T.slots + s.slot0 + i)];
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (int i = tid; i < total; i += kThreads) {
    const uint32_t r = rank_of(i, j);
    const double* src = st + j * c.n;
    const uint32_t* list = T.list + c.list0 + (i - j * c.n);
    const double before = lam[r];
    double acc = 0.0;
    for (int e0 = 0; e0 < c.width; e0 += kAhead) {  // width: a multiple of kAhead
      uint32_t e[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) e[u] = __ldg(list + int64_t(e0 + u) * c.n);
#pragma unroll
      for (int u = 0; u < kAhead; ++u)
        if (e[u] < pad) acc = fma(hop[e[u] >> 16], src[e[u] & 0xffffu], acc);
    }
    lam[r] = before + acc;
  }
}
}  // namespace

int hop_width(int w) { return (w + kAhead - 1) / kAhead * kAhead; }
cudaError_t hop_set_limits() {
  return cudaFuncSetAttribute(k_hop_blocks, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (kHopStates + kHopSlots) * 8);
}

cudaError_t hop_hpsi(const InstDesc& d, const HopPlan& p, double* tab, const double* psi, double* lam,
                     cudaStream_t stream) {
  const unsigned size = 1u << d.lo_bits;
  k_hop_tables<<<dim3((size + 255) / 256, unsigned(2 + d.n - d.lo_bits)), 256, 0, stream>>>(p.diag, d.n, d.lo_bits,
                                                                                            d.vals, tab);
  k_hop_diag<<<stream_grid(d.D), 256, 0, stream>>>(d.sector, d.D, d.lo_bits, p.diag.slot >= 0 ? 1 : 0, tab, psi, lam);
  for (const HopStep& s : p.steps)
    k_hop_blocks<<<unsigned(s.ctas), kThreads, size_t(s.most + s.slots) * 8, stream>>>(
        p.tables, s, d.rank_hi, d.rank_lo, d.lo_bits, d.vals, psi, lam);
  return cudaGetLastError();
}

}  // namespace vqe
