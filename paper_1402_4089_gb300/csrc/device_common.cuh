// Device-side building blocks shared by the kernels of libhmc (sm_103a):
// mbarrier waits with an iteration bound, bulk asynchronous copies, cluster
// (DSMEM) addressing and signalling, and the Philox4x64-10 generator.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_fp16.h>

namespace hmc {

// Error bits written to the handle's device error word.
enum : int {
  ERR_TIMEOUT_STAGE = 1,     // wait for an X tile in shared memory ran out
  ERR_TIMEOUT_EXCHANGE = 2,  // wait for peers' partial logits ran out
  ERR_TIMEOUT_SLOT = 4,      // wait for an exchange slot to be released ran out
  ERR_TIMEOUT_MMA = 8,       // wait for a tensor-core commit ran out
  ERR_BAD_LABEL = 16,        // label outside [0, K)
  ERR_NONFINITE_X = 32,      // non-finite predictor value
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init_cluster() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive_local(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// One probe of the phase with the given parity (CTA-scope acquire).
__device__ __forceinline__ bool mbar_test_cta(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// The same without the short suspension of a phase that is not complete: a look ahead,
// issued before work that need not wait for its answer.
__device__ __forceinline__ bool mbar_look_cta(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// One probe with cluster-scope acquire (data written by peer CTAs).
__device__ __forceinline__ bool mbar_test_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded waits: return false when `limit` probes did not see the phase.
__device__ __forceinline__ bool mbar_wait_cta(uint64_t* bar, uint32_t parity, long long limit) {
  const uint32_t a = smem_u32(bar);
  for (long long i = 0; i < limit; ++i)
    if (mbar_test_cta(a, parity)) return true;
  return false;
}

__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, long long limit) {
  const uint32_t a = smem_u32(bar);
  for (long long i = 0; i < limit; ++i)
    if (mbar_test_cluster(a, parity)) return true;
  return false;
}

// Waits until a copy or an MMA in flight has landed, before shared memory or TMEM is
// released.  Does not give up on an abort, nor at a short spin limit: the caller's limit
// says how long the kernel waits for its work, and what is in flight then still lands.
constexpr long long kDrainProbes = 1ll << 20;
__device__ __forceinline__ void wait_drain(uint64_t* bar, uint32_t parity, long long limit) {
  const uint32_t a = smem_u32(bar);
  const long long n = limit > kDrainProbes ? limit : kDrainProbes;
  for (long long i = 0; i < n; ++i)
    if (mbar_test_cta(a, parity)) return;
}

// A position in a ring of mbarriers: the slot and the parity of its current use.
// Counted, not divided: a 64-bit division by a run-time ring size in front of
// every wait costs the issuing warps more than the waits themselves.
struct Ring {
  int slot = 0;
  uint32_t par = 0;
  __device__ __forceinline__ void next(int n) {
    if (++slot == n) {
      slot = 0;
      par ^= 1u;
    }
  }
};

// ------------------------------------------------------------ launches that overlap
// A kernel launched by launch_chained starts while the kernel before it in the stream
// runs its last blocks, if that one has called chain_next; it calls chain_wait before it
// touches anything that an earlier kernel writes or reads (there the kernels before it are
// complete and their writes visible).  chain_next comes after chain_wait, so a kernel
// that has started knows everything before its direct predecessor to be complete.
// Only the short kernels of the FP32 tensor-core chain call chain_next: the passes start
// under them (barriers, TMEM, the first copies of X).  The long passes do not: with the
// next kernel's blocks waiting on their SMs a gradient at n=1e4 p=5000 C=9 took 98.5 us
// instead of 94.5 (96.2 with no overlap at all), n=6e4 p=785 C=9 152 instead of 150 us.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Given>
inline cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                  Given... given) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, Params(given)...);
}

// ------------------------------------------------------------ exact sums
// Knuth's two-sum: a + b rounded, and what the rounding lost.
__device__ __forceinline__ float two_sum(float a, float b, float& lost) {
  const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
  lost = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return s;
}

// ------------------------------------------------------------ bulk copies
// Contiguous global -> shared copy completing on a local mbarrier
// (both addresses 16-byte aligned, bytes a multiple of 16).
__device__ __forceinline__ void bulk_g2s(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(smem_dst)),
      "l"(gsrc), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// L2 eviction policies, and the copy above under one of them.
__device__ __forceinline__ uint64_t l2_evict_last() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void bulk_g2s_hint(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar,
                                              uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_u32(smem_dst)),
      "l"(gsrc), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// Order this thread's generic-proxy shared-memory writes before later async-proxy reads.
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Four E4M3 values (bytes of w, byte 0 first) -> four BF16 values as two bf16x2
// words (element 0 in the low half of lo).  Exact: the sign to bit 15 and the seven
// bits of exponent and significand to bits 10..4 give a BF16 number 2^120 too small
// (exponent bias 127 for 7; E4M3 subnormals and zero become BF16 ones), and the
// product with 2^120 is exact.  Five instructions a pair; by way of FP16 (hardware
// conversion, fields moved, zeros masked) it took eleven.
__device__ __forceinline__ uint32_t e4m3x2_scaled(uint32_t t) {   // codes in bits 15..8 and 31..24
  return (t & 0x80008000u) | ((t >> 4) & 0x07f007f0u);
}
__device__ __forceinline__ uint32_t bf16x2_mul(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ void fp8x4_to_bf16x4(uint32_t w, uint32_t& lo, uint32_t& hi) {
  constexpr uint32_t k2p120 = 0x7b807b80u;
  lo = bf16x2_mul(e4m3x2_scaled(__byte_perm(w, 0u, 0x1404)), k2p120);
  hi = bf16x2_mul(e4m3x2_scaled(__byte_perm(w, 0u, 0x3424)), k2p120);
}

// Bulk prefetch of a contiguous global range into L2 (16-byte aligned address,
// bytes a multiple of 16); no shared memory and no completion to wait for.
__device__ __forceinline__ void bulk_prefetch_l2(const void* gsrc, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(gsrc), "r"(bytes) : "memory");
}

// ----------------------------------------------------------------- cluster
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_peer(uint32_t local_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
  return r;
}

// Asynchronous remote stores that complete transaction bytes on the remote
// CTA's mbarrier (both addresses already mapped to the peer).
__device__ __forceinline__ void st_async_v4f(uint32_t raddr, float a, float b, float c, float d, uint32_t rbar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(raddr),
      "f"(a), "f"(b), "f"(c), "f"(d), "r"(rbar)
      : "memory");
}

__device__ __forceinline__ void st_async_v2d(uint32_t raddr, double a, double b, uint32_t rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(raddr),
               "d"(a), "d"(b), "r"(rbar)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive_remote(uint32_t rbar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(rbar) : "memory");
}

// --------------------------------------------------------- Philox4x64-10
// Counter-based generator of Salmon, Moraes, Dror & Shaw (SC'11): ten rounds
// of two 64x64->128 multiplies, key bumped by the Weyl constants.
struct u64x4 {
  uint64_t x, y, z, w;
};

__device__ __forceinline__ u64x4 philox4x64_10(u64x4 c, uint64_t k0, uint64_t k1) {
  const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
  const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += W0;
      k1 += W1;
    }
    const uint64_t hi0 = __umul64hi(M0, c.x), lo0 = M0 * c.x;
    const uint64_t hi1 = __umul64hi(M1, c.z), lo1 = M1 * c.z;
    c = u64x4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
  }
  return c;
}

// 64-bit word -> double in (0, 1): ((w >> 11) + 0.5) * 2^-53.
__device__ __forceinline__ double word_to_uniform(uint64_t w) {
  return (static_cast<double>(w >> 11) + 0.5) * 1.1102230246251565404e-16;
}

enum : uint64_t { TAG_MOMENTUM = 0, TAG_ACCEPT = 1 };

// Normals q = 4*blk .. 4*blk+3 of the momentum draw of (chain, iteration):
// Box-Muller on the word pairs (w0, w1) and (w2, w3), cosine then sine.
__device__ __forceinline__ void momentum_block(uint64_t seed, uint64_t iteration, uint64_t chain, uint64_t blk,
                                               double out[4]) {
  const u64x4 w = philox4x64_10(u64x4{blk, iteration, chain, TAG_MOMENTUM}, seed, 0ull);
  const double two_pi = 2.0 * 3.14159265358979323846;
  {
    const double r = sqrt(-2.0 * log(word_to_uniform(w.x)));
    const double t = two_pi * word_to_uniform(w.y);
    out[0] = r * cos(t);
    out[1] = r * sin(t);
  }
  {
    const double r = sqrt(-2.0 * log(word_to_uniform(w.z)));
    const double t = two_pi * word_to_uniform(w.w);
    out[2] = r * cos(t);
    out[3] = r * sin(t);
  }
}

__device__ __forceinline__ double accept_uniform(uint64_t seed, uint64_t iteration, uint64_t chain) {
  const u64x4 w = philox4x64_10(u64x4{0ull, iteration, chain, TAG_ACCEPT}, seed, 0ull);
  return word_to_uniform(w.x);
}

}  // namespace hmc
