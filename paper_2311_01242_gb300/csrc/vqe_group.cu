// Gate sweeps of large real instances (Sec. 2.1.2's rotations and the adjoint gradient
// g_k = 2 <lambda|A_k|phi_k>) in groups of consecutive gates, one launch per group.
//
// The gates of a group touch the qubits of a set S only, so the amplitudes fall into
// independent blocks, one per occupation pattern of the other qubits. A block (at most
// kGroupStates amplitudes) is loaded into shared memory once, all gates of the group
// rotate it there, and it is stored once. Blocks with the same electron counts left for
// S share one list of local states and one pair list per gate, so those lists are small
// and stay in L2; a pair's sign is its local part times the parity of the pattern.
//
// What bounds it and why this form: a launch per gate costs 2 us (forward) to 5 us
// (reverse) at 24 qubits however little the gate does, and reads 8 bytes of pair list
// per pair; 256 gates took 2.2 ms there. A group of 5 to 6 random double excitations (18
// pair gates of a boson sector) costs a launch, about 4 us of tables, loads and stores,
// and per gate shared-memory accesses, 32-bit integer multiply-adds (Q1.62 fixed point:
// two FP64 operations per clock and SM would take longer) and a block barrier: 0.93 ms
// at 24 qubits; 2.7 million boson states and 144 gates 4.6 -> 2.6 ms. Issue slots
// bound the gates of large sectors, latencies the rest. The reverse sweep un-applies psi
// beside lambda ({psi, lambda} as 16 bytes), so no forward outputs are kept; gradient
// sums are integers: exact and independent of the order of blocks (cross_add). Tried: 256
// threads per CTA (24 qubits 8 % slower), 608 CTAs (10 % slower, nothing of the next launch
// fits beside them), 5,120 amplitudes per CTA (boson sector 10 % slower), pair lists read
// from L2 gate by gate (a latency per gate).
#include <climits>
#include <cuda_runtime.h>

#include "vqe_internal.h"
#include "vqe_device.cuh"

namespace vqe {
namespace {

constexpr int kWarps = kGroupThreads / 32;
constexpr int kBatch = 8;  // independent loads per thread

__device__ __forceinline__ void pdl_wait_release() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void copy8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// psi = |HF>, the gates' cos and sin in fixed point (spread over the blocks: sincos
// runs on the FP64 pipe), gradient sums 0; *bad becomes non-zero if an angle of a gate
// with pairs is not finite.
__global__ void __launch_bounds__(kStreamThreads)
k_group_init(int64_t D, int64_t hf_rank, int M, const int64_t* __restrict__ pair_off,
             const double* __restrict__ theta, long long* __restrict__ psi, int4* __restrict__ trig,
             unsigned long long* __restrict__ gacc, int* __restrict__ bad) {
  const int64_t i0 = blockIdx.x * int64_t(blockDim.x) + threadIdx.x, step = int64_t(gridDim.x) * blockDim.x;
  for (int m = int(blockIdx.x) + int(threadIdx.x) * int(gridDim.x); m < M; m += int(step)) {
    double s, c;
    sincos(theta[m], &s, &c);
    if (!(fabs(c) <= 1.0) && __ldg(pair_off + m + 1) > __ldg(pair_off + m)) *bad = 1;
    trig[m] = fixed_trig(c, s);
  }
  for (int64_t r = i0; r < D; r += step) psi[r] = r == hf_rank ? 1ll << 62 : 0ll;
  if (gacc)
    for (int64_t r = i0; r < int64_t(M) * 2 * kGroupCopies; r += step) gacc[r] = 0ull;
}

struct GateShared {
  int ch, cl, sh, sl;
  int first, n;        // pairs of one block
  uint32_t inv;        // 2^32 / n, rounded up
};

// One group on one CTA's blocks. v: psi, or {psi, lambda}.
template <bool REV>
__global__ void __launch_bounds__(kGroupThreads, 2)
k_group_gates(const GroupTables T, const GroupStep s, long long* __restrict__ v, const int4* __restrict__ trig,
              unsigned long long* __restrict__ gacc, int M, int store) {
  extern __shared__ __align__(16) long long st[];
  __shared__ GateShared gate[kGroupGates];
  __shared__ uint32_t sign[kGroupPatterns];  // of each block, a bit per gate
  __shared__ long long part[REV ? kGroupGates * kWarps : 1];
  __shared__ uint32_t part_lo[REV ? kGroupGates * kWarps : 1];
  longlong2* st2 = reinterpret_cast<longlong2*>(st);
  uint32_t* pairs = reinterpret_cast<uint32_t*>(st + size_t(s.most) * (REV ? 2 : 1));
  uint32_t* rank = pairs + s.most_pairs;
  longlong2* v2 = reinterpret_cast<longlong2*>(v);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const GroupWork w = T.work[s.work0 + blockIdx.x];
  const GroupClass c = T.classes[w.cls];
  const uint32_t st_a = uint32_t(__cvta_generic_to_shared(st)), lo_mask = (1u << T.lo_bits) - 1u;
  const int total = c.n * w.count;
  // everything that does not depend on the launches before
  const uint32_t pairs_a = uint32_t(__cvta_generic_to_shared(pairs));
  for (int i = tid * 4; i < c.pairs; i += kGroupThreads * 4) copy16(pairs_a + uint32_t(i) * 4u, T.pairs + c.pair0 + i);
  for (int i = tid; i < w.count; i += kGroupThreads) {
    const uint32_t k = __ldg(T.patterns + w.first + i);
    uint32_t b = 0;
    for (int g = 0; g < s.gates; ++g) b |= uint32_t(parity32(k & __ldg(&T.gates[s.gate0 + g].par))) << g;
    sign[i] = b;
  }
  for (int i0 = tid; i0 < total; i0 += kGroupThreads * kBatch) {
    uint32_t k[kBatch], hi[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int i = min(i0 + u * kGroupThreads, total - 1);
      const int j = c.n == total ? 0 : int(__umulhi(uint32_t(i), c.inv));
      k[u] = __ldg(T.states + c.state0 + i - j * c.n);
      hi[u] = __ldg(T.patterns + w.first + j);
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const uint32_t v = k[u] | hi[u];
      hi[u] = __ldg(T.rank_hi + (v >> T.lo_bits));
      k[u] = __ldg(T.rank_lo + (v & lo_mask));
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (i0 + u * kGroupThreads < total) rank[i0 + u * kGroupThreads] = hi[u] + k[u];
  }
  GroupGate rec{};
  int2 range = make_int2(0, 0);
  if (tid < s.gates) {
    rec = T.gates[s.gate0 + tid];
    range = __ldg(T.ranges + c.range0 + tid);
  }
  pdl_wait_release();
#pragma unroll 4
  for (int i = tid; i < total; i += kGroupThreads) {  // the same thread's ranks
    if (REV)
      copy16(st_a + uint32_t(i) * 16u, v2 + rank[i]);
    else
      copy8(st_a + uint32_t(i) * 8u, v + rank[i]);
  }
  if (tid < s.gates) {
    const int4 t = trig[rec.m];
    gate[tid] = GateShared{t.x, t.y, t.z, t.w, range.x, range.y,
                           range.y > 1 ? 0xffffffffu / uint32_t(range.y) + 1u : 0u};
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int g0 = REV ? s.gates - 1 : 0, step = REV ? -1 : 1;
  GateShared t = gate[g0];
  for (int k = 0; k < s.gates; ++k) {
    CrossSum acc{0, 0u};
    const int n = t.n * w.count, g = g0 + k * step;
    const int nh = -t.sh, nl = -t.sl;
#pragma unroll 1
    for (int q = tid; q < n; q += kGroupThreads) {
      const int j = t.inv ? int(__umulhi(uint32_t(q), t.inv)) : q;
      const uint32_t e = pairs[t.first + (q - j * t.n)];
      const bool swap = ((sign[j] >> g) & 1u) != 0;  // a pair of the other sign turns the other way
      const int i0 = j * c.n + int(e & 0xffffu), i1 = j * c.n + int(e >> 16);
      const int ia = swap ? i1 : i0, ib = swap ? i0 : i1;
      if (REV) {
        const longlong2 va = st2[ia], vb = st2[ib];
        const Words a = split(va.x), b = split(vb.x), la = split(va.y), lb = split(vb.y);
        st2[ia] = make_longlong2(turn(a, b, t.ch, t.cl, t.sh, t.sl), turn(la, lb, t.ch, t.cl, t.sh, t.sl));
        st2[ib] = make_longlong2(turn(b, a, t.ch, t.cl, nh, nl), turn(lb, la, t.ch, t.cl, nh, nl));
        cross_add(acc, a, lb, b, la, false);
      } else {
        const Words a = split(st[ia]), b = split(st[ib]);
        st[ia] = turn(a, b, t.ch, t.cl, nh, nl);
        st[ib] = turn(b, a, t.ch, t.cl, t.sh, t.sl);
      }
    }
    if (k + 1 < s.gates) t = gate[g + step];
    if (REV) {
      if ((tid & ~31) < n) acc = cross_warp(acc);
      if (lane == 0) {
        part[g * kWarps + warp] = acc.hi;
        part_lo[g * kWarps + warp] = acc.lo;
      }
    }
    if (n > 0) __syncthreads();
  }
  if (REV) {
    __syncthreads();
    if (tid < s.gates && range.y > 0) {
      long long r = 0;
      unsigned long long lo = 0;
#pragma unroll
      for (int i = 0; i < kWarps; ++i) {
        r += part[tid * kWarps + i];
        lo += part_lo[tid * kWarps + i];
      }
      unsigned long long* to = gacc + int64_t(blockIdx.x % kGroupCopies) * 2 * M + rec.m;
      atomicAdd(to, static_cast<unsigned long long>(r));
      atomicAdd(to + M, lo);
    }
  }
  if (!store) return;
#pragma unroll 4
  for (int i = tid; i < total; i += kGroupThreads) {
    if (REV)
      v2[rank[i]] = st2[i];
    else
      v[rank[i]] = st[i];
  }
}

// psi from fixed point to FP64 in place; NaN after an angle that is not finite
__global__ void __launch_bounds__(kStreamThreads)
k_group_out(int64_t D, const int* __restrict__ bad, double* __restrict__ psi) {
  const double nan = llbits(0x7ff8000000000000ll);
  const bool lost = *bad != 0;
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < D; r += int64_t(gridDim.x) * blockDim.x)
    psi[r] = lost ? nan : __ll2double_rn(__double_as_longlong(psi[r])) * 0x1p-62;
}

// {psi, lambda} in fixed point, lambda below 2^61
__global__ void __launch_bounds__(kStreamThreads)
k_group_in(int64_t D, const double* __restrict__ l2, const double* __restrict__ psi, const double* __restrict__ lam,
           longlong2* __restrict__ v) {
  const double sc = pow2(61 - norm_exp(*l2));
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < D; r += int64_t(gridDim.x) * blockDim.x)
    v[r] = make_longlong2(__double2ll_rn(psi[r] * 0x1p62), __double2ll_rn(lam[r] * sc));
}

// per-block partials of <lambda|lambda>, and their sum in a fixed order
__global__ void __launch_bounds__(kStreamThreads)
k_group_norm(const double* __restrict__ lam, int64_t D, double* __restrict__ part) {
  __shared__ double red[32];
  double v = 0.0;
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < D; r += int64_t(gridDim.x) * blockDim.x)
    v = fma(lam[r], lam[r], v);
  v = block_sum(v, red);
  if (threadIdx.x == 0) part[blockIdx.x] = v;
}
__global__ void __launch_bounds__(kStreamThreads) k_group_norm_sum(const double* __restrict__ part, int n,
                                                                   double* __restrict__ l2) {
  __shared__ double red[32];
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += kStreamThreads) v += part[i];
  v = block_sum(v, red);
  if (threadIdx.x == 0) *l2 = v;
}

// gradients; NaN where lambda is not finite
__global__ void __launch_bounds__(kStreamThreads)
k_group_final(const unsigned long long* __restrict__ gacc, int M, const double* __restrict__ l2,
              double* __restrict__ grad) {
  const int m = blockIdx.x * kStreamThreads + threadIdx.x;
  if (m >= M) return;
  unsigned long long v = 0, lo = 0;
#pragma unroll 8
  for (int i = 0; i < kGroupCopies; ++i) {
    v += gacc[int64_t(2 * i) * M + m];
    lo += gacc[int64_t(2 * i + 1) * M + m];
  }
  const double n2 = *l2;
  grad[m] = n2 < llbits(0x7ff0000000000000ll)
                ? cross_value(static_cast<long long>(v), lo) * pow2(norm_exp(n2) - 61)
                : llbits(0x7ff8000000000000ll);
}

template <bool REV>
cudaError_t launch(const GroupTables& t, const GroupStep& s, long long* v, const GroupBuffers& w, int M, int store,
                   cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(s.ctas));
  cfg.blockDim = dim3(kGroupThreads);
  cfg.dynamicSmemBytes = size_t(s.most) * (REV ? 20 : 12) + size_t(s.most_pairs) * 4;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_group_gates<REV>, t, s, v, static_cast<const int4*>(w.trig), w.gacc, M, store);
}
}  // namespace

cudaError_t group_set_limits() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(k_group_gates<false>, a, kGroupStates * 12 + (kGroupPairs + 4) * 4);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(k_group_gates<true>, a, kGroupStates * 20 + (kGroupPairs + 4) * 4);
}

cudaError_t group_forward(const InstDesc& d, const GroupPlan& p, const GroupBuffers& w, const double* theta,
                          double* psi, bool with_grad, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(w.bad, 0, sizeof(int), stream);
  if (e != cudaSuccess) return e;
  k_group_init<<<stream_grid(d.D), kStreamThreads, 0, stream>>>(d.D, d.hf_rank, d.M, d.pair_off, theta,
                                                                reinterpret_cast<long long*>(psi), w.trig,
                                                                with_grad ? w.gacc : nullptr, w.bad);
  for (const GroupStep& s : p.steps)
    if ((e = launch<false>(p.tables, s, reinterpret_cast<long long*>(psi), w, d.M, 1, stream)) != cudaSuccess) return e;
  k_group_out<<<stream_grid(d.D), kStreamThreads, 0, stream>>>(d.D, w.bad, psi);
  return cudaGetLastError();
}

cudaError_t group_reverse(const InstDesc& d, const GroupPlan& p, const GroupBuffers& w, const double* psi,
                          const double* lam, void* scratch, double* grad, cudaStream_t stream) {
  const int grid = stream_grid(d.D);
  k_group_norm<<<grid, kStreamThreads, 0, stream>>>(lam, d.D, w.norm + 1);
  k_group_norm_sum<<<1, kStreamThreads, 0, stream>>>(w.norm + 1, grid, w.norm);
  k_group_in<<<grid, kStreamThreads, 0, stream>>>(d.D, w.norm, psi, lam, static_cast<longlong2*>(scratch));
  for (size_t i = p.steps.size(); i-- > 0;) {
    const cudaError_t e =
        launch<true>(p.tables, p.steps[i], static_cast<long long*>(scratch), w, d.M, i > 0 ? 1 : 0, stream);
    if (e != cudaSuccess) return e;
  }
  if (d.M > 0)
    k_group_final<<<(d.M + kStreamThreads - 1) / kStreamThreads, kStreamThreads, 0, stream>>>(w.gacc, d.M, w.norm,
                                                                                              grad);
  return cudaGetLastError();
}

}  // namespace vqe
