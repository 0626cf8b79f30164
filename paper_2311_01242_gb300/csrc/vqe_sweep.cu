// Gate sweeps of mid-size real instances (spin sectors of 256 to 131,072 states), for one
// instance or a batch: the forward sweep and the reverse sweep with the gradient
// (Sec. 2.1.2's rotations, g_k = 2 <lambda|A_k|phi_k>) as one launch each, a
// thread-block cluster per instance with the state in the cluster's shared memory.
// H psi runs between them on the tensor cores (vqe_tc.cu).
//
// What bounds a gate and why this form: a gate has only a few hundred to a few
// thousand pairs and every gate depends on the one before. As a launch per gate it
// costs 2 us (forward) to 4 us (reverse) whatever its size. Here a gate costs its
// chain: a pair's two amplitudes from (distributed) shared memory, the rotation, the
// stores and one barrier. Amplitudes are 64-bit fixed point as in the resident
// kernel (Q1.62; lambda below its norm), because a rotation is 12 32-bit multiply-adds
// on the integer pipe against four FP64 ones at two per clock and SM. The forward sweep streams each pair's two
// outputs, phi at that gate, to the workspace (coalesced, 16 bytes per pair), so the
// reverse sweep keeps lambda only. Gradient contributions are summed as integers:
// exact, so no result depends on the cluster size or on any order (16 bits of each product
// below the fixed point's unit are summed beside it: 735 -> 742 us at 16 qubits and 360
// angles, nothing at 20 qubits; without them the gradient lost up to a digit).
#include <climits>
#include <cuda_runtime.h>

#include "vqe_internal.h"
#include "vqe_device.cuh"

namespace vqe {
namespace {

constexpr int kMaxThreads = 512;
constexpr int kAhead = 2;   // pairs per thread copied ahead
constexpr int kSlots = 5;   // gates in the ring: this one and the next four
constexpr int kDots = kSweepDots;

// cos and sin as 62-bit fixed point in two signed words, x = (h 2^32 + l) 2^-62
struct GateTab {
  int32_t ch, cl, sh, sl;
  int32_t lo, n;  // this CTA's pairs
  int32_t pad0, pad1;
};

template <int C>
struct Cluster {
  static __device__ __forceinline__ uint32_t rank() {
    if constexpr (C == 1) return 0u;
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
  }
  // every thread of the cluster; orders shared-memory accesses across it
  static __device__ __forceinline__ void sync() {
    if constexpr (C == 1) {
      __syncthreads();
    } else {
      asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  }
  // amplitude r lives in CTA r >> shift
  static __device__ __forceinline__ uint32_t addr(uint32_t base, uint32_t r, int shift) {
    if constexpr (C == 1) return base + r * 8u;
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(a)
                 : "r"(base + (r & ((1u << shift) - 1u)) * 8u), "r"(r >> shift));
    return a;
  }
  static __device__ __forceinline__ long long ld(uint32_t a) {
    long long v;
    if constexpr (C == 1)
      asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    else
      asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
  }
  static __device__ __forceinline__ void st(uint32_t a, long long v) {
    if constexpr (C == 1)
      asm volatile("st.shared.b64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
    else
      asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
  }
};

// A batch's launches for the other cluster sizes follow each other with programmatic
// dependent launch and depend on nothing of each other: the next may start at once,
// and each ends after the one before, so the last one's end is everyone's.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Copies of a thread's own pair inputs into the ring, read back by the same thread
// (asynchronous copies: registers loaded that far ahead share scoreboards, and
// waiting for the oldest then waits for all, one memory latency per gate).
__device__ __forceinline__ void copy8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ unsigned long long clock_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The batch's wait check (vqe_batch_set_wait): the probed task waits for a count
// that nothing reaches, for at most the budget, then records itself in the status
// word; the outputs of every instance swept here or in the persistent launch become NaN.
__device__ __forceinline__ void probe_wait(const SweepCtl& ctl, int task) {
  if (task != ctl.probe || threadIdx.x != 0) return;
  const unsigned long long t0 = clock_ns();
  for (long long it = 0; it < ctl.budget_ns / 64 + 1024; ++it) {
    if (*static_cast<const volatile int*>(ctl.never) != 0) return;
    __nanosleep(256);
    if (static_cast<long long>(clock_ns() - t0) > ctl.budget_ns) break;
  }
  atomicCAS(ctl.status, 0, task + 1);
}

template <int C>
__device__ __forceinline__ void fill_table(GateTab* tab, const int64_t* pair_off, int M, uint32_t rank,
                                           const double* th) {
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    double s, c;
    sincos(th[m], &s, &c);
    const int64_t p0 = __ldg(pair_off + m), n = __ldg(pair_off + m + 1) - p0;
    const int64_t lo = n * rank / C, hi = n * (rank + 1) / C;
    GateTab t;
    const int4 f = fixed_trig(c, s);
    t.ch = f.x;
    t.cl = f.y;
    t.sh = f.z;
    t.sl = f.w;
    t.lo = int32_t(p0 + lo);
    t.n = int32_t(hi - lo);
    tab[m] = t;
  }
}

// Forward sweep. The gate loop is bound by issue (about 75 instructions per pair and
// warp, and what every warp does per gate) and by the chain load, multiply, store,
// barrier; a pair entry's load takes longer than a small gate, so entries are copied to
// shared memory four gates ahead.
template <int C>
__global__ void __launch_bounds__(kMaxThreads, 1)
k_sweep_fwd(const SweepInst* __restrict__ many, const SweepInst one, char* ws, const double* __restrict__ theta,
            int64_t ld_theta, int keep, const SweepCtl ctl) {
  extern __shared__ __align__(16) unsigned char smem[];
  typedef Cluster<C> K;
  const SweepInst* I = many ? many + int(blockIdx.x) / C : &one;
  const uint32_t rank = K::rank();
  const int tid = threadIdx.x, T = blockDim.x, cap = kAhead * T, M = I->M, shift = I->shift, D = I->D;
  const uint2* __restrict__ pairs = I->rpairs;
  GateTab* tab = reinterpret_cast<GateTab*>(smem);
  uint2* ring = reinterpret_cast<uint2*>(tab + M);
  const uint32_t ring_a = uint32_t(__cvta_generic_to_shared(ring));
  long long* st = reinterpret_cast<long long*>(ring + kSlots * cap);
  const uint32_t base = uint32_t(__cvta_generic_to_shared(st));
  longlong2* __restrict__ phi = reinterpret_cast<longlong2*>(ws + I->phi);
  pdl_release();
  if (ctl.probe >= 0 && rank == 0) probe_wait(ctl, ctl.task0 + I->task);
  fill_table<C>(tab, I->pair_off, M, rank, theta + I->inst * ld_theta);
  const int mine = C == 1 ? D : 1 << shift;
  for (int r = tid; r < mine; r += T) st[r] = 0;
  if (rank == 0) {
    unsigned long long* g = reinterpret_cast<unsigned long long*>(ws + I->gacc);
    for (int m = tid; m < 2 * M; m += T) g[m] = 0ull;  // high parts, then low parts
  }
  K::sync();
  if (rank == 0 && tid == 0) K::st(K::addr(base, uint32_t(I->hf_rank), shift), 1ll << 62);
  K::sync();

  auto ahead = [&](int m, int slot) {
    if (m < M) {
      const int lo = tab[m].lo, n = tab[m].n;
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int q = tid + u * T;
        if (q < n) copy8(ring_a + uint32_t(slot * cap + q) * 8u, pairs + lo + q);
      }
    }
    copy_commit();
  };
#pragma unroll
  for (int k = 0; k < kSlots - 1; ++k) ahead(k, k);
  copy_wait<kSlots - 2>();
  int slot = 0;
  GateTab t = tab[0];
  uint2 e[kAhead];
#pragma unroll
  for (int u = 0; u < kAhead; ++u) e[u] = M > 0 && tid + u * T < t.n ? ring[tid + u * T] : make_uint2(0u, 0u);
  for (int m = 0; m < M; ++m) {
    // every load of the gate, then what can overlap it (the copies gates ahead),
    // then its arithmetic and stores (a gate's pairs are disjoint); the next gate's
    // record and entries are read before the barrier
    uint32_t xa[kAhead], xb[kAhead];
    long long a[kAhead], b[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (tid + u * T < t.n) {
        xa[u] = K::addr(base, e[u].x & 0x7fffffffu, shift);
        xb[u] = K::addr(base, e[u].y, shift);
        a[u] = K::ld(xa[u]);
        b[u] = K::ld(xb[u]);
      }
    ahead(m + kSlots - 1, slot == 0 ? kSlots - 1 : slot - 1);
    auto rotate = [&](uint32_t px, uint32_t ya, uint32_t yb, long long va, long long vb, int q) {
      const bool neg = int(px) < 0;  // the pair's sign
      const int sh = neg ? -t.sh : t.sh, sl = neg ? -t.sl : t.sl;
      const Words wa = split(va), wb = split(vb);
      const long long na = turn(wa, wb, t.ch, t.cl, -sh, -sl);
      const long long nb = turn(wb, wa, t.ch, t.cl, sh, sl);
      K::st(ya, na);
      K::st(yb, nb);
      if (keep) __stcg(phi + t.lo + q, make_longlong2(na, nb));
    };
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (tid + u * T < t.n) rotate(e[u].x, xa[u], xb[u], a[u], b[u], tid + u * T);
    for (int q = tid + cap; q < t.n; q += T) {
      const uint2 pr = __ldg(pairs + t.lo + q);
      const uint32_t ya = K::addr(base, pr.x & 0x7fffffffu, shift), yb = K::addr(base, pr.y, shift);
      rotate(pr.x, ya, yb, K::ld(ya), K::ld(yb), q);
    }
    if constexpr (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    slot = slot == kSlots - 1 ? 0 : slot + 1;
    copy_wait<kSlots - 2>();
    if (m + 1 < M) {
      t = tab[m + 1];
#pragma unroll
      for (int u = 0; u < kAhead; ++u)
        if (tid + u * T < t.n) e[u] = ring[slot * cap + tid + u * T];
    }
    if constexpr (C > 1)
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else
      __syncthreads();
  }
  // psi in alpha-major order for H psi
  double* psi_am = reinterpret_cast<double*>(ws + I->psi_am);
  const uint32_t* perm = I->perm;
  for (int i = int(rank) * T + tid; i < D; i += C * T)
    psi_am[i] = __ll2double_rn(K::ld(K::addr(base, __ldg(perm + i), shift))) * 0x1p-62;
  K::sync();  // no CTA leaves while its amplitudes are read
  pdl_wait();
}

// Fixed partial sums of psi . lambda and lambda . lambda (alpha-major).
__global__ void __launch_bounds__(256) k_sweep_dot(const SweepInst* __restrict__ many, const SweepInst one, char* ws) {
  __shared__ double red[32];
  const SweepInst& I = many ? many[blockIdx.y] : one;
  const double* psi = reinterpret_cast<const double*>(ws + I.psi_am);
  const double* lam = reinterpret_cast<const double*>(ws + I.lam_am);
  double e = 0.0, l2 = 0.0;
  for (int i = int(blockIdx.x) * 256 + int(threadIdx.x); i < I.D; i += kDots * 256) {
    const double l = lam[i];
    e = fma(psi[i], l, e);
    l2 = fma(l, l, l2);
  }
  e = block_sum(e, red);
  l2 = block_sum(l2, red);
  if (threadIdx.x == 0) {
    double* out = reinterpret_cast<double*>(ws + I.dot) + 2 * blockIdx.x;
    out[0] = e;
    out[1] = l2;
  }
}

// Sum of one of the two columns of partials, in a fixed order.
__device__ __forceinline__ double dot_total(const char* ws, const SweepInst& I, int which) {
  const double* p = reinterpret_cast<const double*>(ws + I.dot) + which;
  double s = 0.0;
  for (int i = 0; i < kDots; ++i) s += p[2 * i];
  return s;
}
// Reverse sweep: gradient contributions from the forward sweep's outputs and lambda,
// then lambda <- U_k^T lambda (inputs copied gates ahead as in the forward sweep).
template <int C>
__global__ void __launch_bounds__(kMaxThreads, 1)
k_sweep_rev(const SweepInst* __restrict__ many, const SweepInst one, char* ws, const double* __restrict__ theta,
            int64_t ld_theta, const SweepCtl ctl) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double scale;
  typedef Cluster<C> K;
  const SweepInst* I = many ? many + int(blockIdx.x) / C : &one;
  const uint32_t rank = K::rank();
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x, cap = kAhead * T, M = I->M, shift = I->shift, D = I->D;
  const uint2* __restrict__ pairs = I->rpairs;
  GateTab* tab = reinterpret_cast<GateTab*>(smem);
  longlong2* fring = reinterpret_cast<longlong2*>(tab + M);
  uint2* ring = reinterpret_cast<uint2*>(fring + kSlots * cap);
  const uint32_t ring_a = uint32_t(__cvta_generic_to_shared(ring));
  const uint32_t fring_a = uint32_t(__cvta_generic_to_shared(fring));
  long long* st = reinterpret_cast<long long*>(ring + kSlots * cap);
  const uint32_t base = uint32_t(__cvta_generic_to_shared(st));
  const longlong2* __restrict__ phi = reinterpret_cast<const longlong2*>(ws + I->phi);
  unsigned long long* gacc = reinterpret_cast<unsigned long long*>(ws + I->gacc);
  pdl_release();
  if (ctl.probe >= 0 && rank == 0) probe_wait(ctl, ctl.task0 + ctl.n + I->task);
  fill_table<C>(tab, I->pair_off, M, rank, theta + I->inst * ld_theta);
  if (tid == 0) scale = pow2(61 - norm_exp(dot_total(ws, *I, 1)));
  K::sync();  // the other CTAs have started: their shared memory may be written
  const double* lam_am = reinterpret_cast<const double*>(ws + I->lam_am);
  const uint32_t* perm = I->perm;
  for (int i = int(rank) * T + tid; i < D; i += C * T)
    K::st(K::addr(base, __ldg(perm + i), shift), __double2ll_rn(lam_am[i] * scale));
  K::sync();

  auto ahead = [&](int m, int slot) {
    if (m >= 0) {
      const int lo = tab[m].lo, n = tab[m].n;
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int q = tid + u * T;
        if (q < n) {
          copy8(ring_a + uint32_t(slot * cap + q) * 8u, pairs + lo + q);
          copy16(fring_a + uint32_t(slot * cap + q) * 16u, phi + lo + q);
        }
      }
    }
    copy_commit();
  };
#pragma unroll
  for (int k = 0; k < kSlots - 1; ++k) ahead(M - 1 - k, k);
  copy_wait<kSlots - 2>();
  int slot = 0;
  GateTab t = tab[M > 0 ? M - 1 : 0];
  uint2 e[kAhead];
  longlong2 f[kAhead];
#pragma unroll
  for (int u = 0; u < kAhead; ++u) {
    const bool in = M > 0 && tid + u * T < t.n;
    e[u] = in ? ring[tid + u * T] : make_uint2(0u, 0u);
    f[u] = in ? fring[tid + u * T] : make_longlong2(0, 0);
  }
  CrossSum acc{0, 0u};
  int counted = 0;  // pairs of the gate that acc belongs to
  auto add_up = [&](int m) {
    if ((tid & ~31) >= counted) return;
    const CrossSum s = cross_warp(acc);  // the same in every lane
    if (lane < 2) atomicAdd(gacc + (lane ? M + m : m), lane ? s.lo : static_cast<unsigned long long>(s.hi));
  };
  for (int m = M - 1; m >= 0; --m) {
    uint32_t xa[kAhead], xb[kAhead];
    long long a[kAhead], b[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (tid + u * T < t.n) {
        xa[u] = K::addr(base, e[u].x & 0x7fffffffu, shift);
        xb[u] = K::addr(base, e[u].y, shift);
        a[u] = K::ld(xa[u]);
        b[u] = K::ld(xb[u]);
      }
    ahead(m - kSlots + 1, slot == 0 ? kSlots - 1 : slot - 1);
    add_up(m + 1);  // of the gate before, while this one's amplitudes arrive
    acc = CrossSum{0, 0u};
    counted = t.n;
    auto step = [&](uint32_t px, longlong2 ph, uint32_t ya, uint32_t yb, long long va, long long vb) {
      const bool neg = int(px) < 0;
      const int sh = neg ? -t.sh : t.sh, sl = neg ? -t.sl : t.sl;
      const Words wa = split(va), wb = split(vb);
      K::st(ya, turn(wa, wb, t.ch, t.cl, sh, sl));
      K::st(yb, turn(wb, wa, t.ch, t.cl, -sh, -sl));
      cross_add(acc, split(ph.x), wb, split(ph.y), wa, neg);
    };
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (tid + u * T < t.n) step(e[u].x, f[u], xa[u], xb[u], a[u], b[u]);
    for (int q = tid + cap; q < t.n; q += T) {
      const uint2 pr = __ldg(pairs + t.lo + q);
      const uint32_t ya = K::addr(base, pr.x & 0x7fffffffu, shift), yb = K::addr(base, pr.y, shift);
      step(pr.x, __ldcg(phi + t.lo + q), ya, yb, K::ld(ya), K::ld(yb));
    }
    if constexpr (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    slot = slot == kSlots - 1 ? 0 : slot + 1;
    copy_wait<kSlots - 2>();
    if (m > 0) {
      t = tab[m - 1];
#pragma unroll
      for (int u = 0; u < kAhead; ++u)
        if (tid + u * T < t.n) {
          e[u] = ring[slot * cap + tid + u * T];
          f[u] = fring[slot * cap + tid + u * T];
        }
    }
    if constexpr (C > 1)
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else
      __syncthreads();
  }
  if (M > 0) add_up(0);
  pdl_wait();
}

// Energies and gradients; NaN where the batch recorded a failed wait, an angle of a
// gate with pairs is not finite (fixed point holds no NaN) or lambda is not.
__global__ void __launch_bounds__(256) k_sweep_final(const SweepInst* __restrict__ many, const SweepInst one,
                                                     const char* ws, const double* __restrict__ theta, int64_t ld_theta,
                                                     const SweepCtl ctl, double* __restrict__ energy,
                                                     double* __restrict__ grad, int64_t ld_grad) {
  const SweepInst& I = many ? many[blockIdx.x] : one;
  const double nan = llbits(0x7ff8000000000000ll);
  int odd = ctl.status && *ctl.status != 0;
  for (int m = threadIdx.x; m < I.M; m += 256)
    odd |= !(fabs(theta[I.inst * ld_theta + m]) < llbits(0x7ff0000000000000ll)) && I.pair_off[m + 1] > I.pair_off[m];
  const bool lost = __syncthreads_or(odd) != 0;
  if (threadIdx.x == 0) energy[I.inst] = lost ? nan : dot_total(ws, I, 0);
  if (!grad) return;
  const double l2 = dot_total(ws, I, 1);
  const bool bad = lost || !(l2 < llbits(0x7ff0000000000000ll));
  const double sc = pow2(norm_exp(l2) - 61);
  const long long* g = reinterpret_cast<const long long*>(ws + I.gacc);
  for (int m = threadIdx.x; m < I.M; m += 256)
    grad[I.inst * ld_grad + m] = bad ? nan : cross_value(g[m], static_cast<unsigned long long>(g[I.M + m])) * sc;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*kernel)(KArgs...), const SweepClass& k, int c, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(k.n * c));
  cfg.blockDim = dim3(unsigned(k.threads));
  cfg.dynamicSmemBytes = k.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(c);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = k.follows ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int C>
cudaError_t fwd(const SweepClass& k, const SweepInst* one, char* ws, const double* theta, int64_t ld, bool keep,
                const SweepCtl& ctl, cudaStream_t s) {
  return launch_cluster(k_sweep_fwd<C>, k, C, s, one ? nullptr : k.insts, one ? *one : SweepInst{}, ws, theta,
                        ld, keep ? 1 : 0, ctl);
}
template <int C>
cudaError_t rev(const SweepClass& k, const SweepInst* one, char* ws, const double* theta, int64_t ld,
                const SweepCtl& ctl, cudaStream_t s) {
  return launch_cluster(k_sweep_rev<C>, k, C, s, one ? nullptr : k.insts, one ? *one : SweepInst{}, ws, theta,
                        ld, ctl);
}
template <int C>
cudaError_t limits(int bytes) {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_sweep_fwd<C>, a, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sweep_rev<C>, a, bytes);
  if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(k_sweep_fwd<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(k_sweep_rev<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}
}  // namespace

size_t sweep_smem(int M, int c, int shift, int64_t D, int threads) {
  return size_t(M) * sizeof(GateTab) + size_t(kSlots) * kAhead * threads * 24 + (c == 1 ? size_t(D) : size_t(1) << shift) * 8;
}

cudaError_t sweep_set_limits(size_t optin) {
  const int b = int(optin) - 1024;  // beside the static arrays
  cudaError_t e = limits<1>(b);
  if (e == cudaSuccess) e = limits<2>(b);
  if (e == cudaSuccess) e = limits<4>(b);
  if (e == cudaSuccess) e = limits<8>(b);
  if (e == cudaSuccess) e = limits<16>(b);
  return e;
}

bool sweep_wide_clusters() {
  static const bool ok = [] {
    int dev = 0, optin = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        sweep_set_limits(size_t(optin)) != cudaSuccess)
      return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kMaxThreads);
    cfg.dynamicSmemBytes = size_t(optin) - 1024;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 16;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool fits = cudaOccupancyMaxActiveClusters(&n, k_sweep_rev<16>, &cfg) == cudaSuccess && n > 0;
    cudaGetLastError();
    return fits;
  }();
  return ok;
}

cudaError_t sweep_forward(const SweepClass& k, const SweepInst* one, char* ws, const double* theta, int64_t ld_theta,
                          bool keep, const SweepCtl& ctl, cudaStream_t s) {
  switch (k.c) {
    case 1: return fwd<1>(k, one, ws, theta, ld_theta, keep, ctl, s);
    case 2: return fwd<2>(k, one, ws, theta, ld_theta, keep, ctl, s);
    case 4: return fwd<4>(k, one, ws, theta, ld_theta, keep, ctl, s);
    case 8: return fwd<8>(k, one, ws, theta, ld_theta, keep, ctl, s);
    default: return fwd<16>(k, one, ws, theta, ld_theta, keep, ctl, s);
  }
}

cudaError_t sweep_dots(const SweepInst* many, const SweepInst* one, int n, char* ws, cudaStream_t s) {
  k_sweep_dot<<<dim3(kDots, unsigned(n)), 256, 0, s>>>(one ? nullptr : many, one ? *one : SweepInst{}, ws);
  return cudaGetLastError();
}

cudaError_t sweep_reverse(const SweepClass& k, const SweepInst* one, char* ws, const double* theta, int64_t ld_theta,
                          const SweepCtl& ctl, cudaStream_t s) {
  switch (k.c) {
    case 1: return rev<1>(k, one, ws, theta, ld_theta, ctl, s);
    case 2: return rev<2>(k, one, ws, theta, ld_theta, ctl, s);
    case 4: return rev<4>(k, one, ws, theta, ld_theta, ctl, s);
    case 8: return rev<8>(k, one, ws, theta, ld_theta, ctl, s);
    default: return rev<16>(k, one, ws, theta, ld_theta, ctl, s);
  }
}

cudaError_t sweep_final(const SweepInst* many, const SweepInst* one, int n, const char* ws, const double* theta,
                        int64_t ld_theta, const SweepCtl& ctl, double* energy, double* grad, int64_t ld_grad,
                        cudaStream_t s) {
  k_sweep_final<<<unsigned(n), 256, 0, s>>>(one ? nullptr : many, one ? *one : SweepInst{}, ws, theta, ld_theta, ctl,
                                            energy, grad, ld_grad);
  return cudaGetLastError();
}

}  // namespace vqe
