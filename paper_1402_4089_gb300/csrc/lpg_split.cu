// Two-pass evaluation of the log-posterior and its gradient for FP32 X on the
// tensor cores (Eqs. softmax, loglike, logkernel and gradient of Sec. 2.1),
// used by the two-pass FP32 engine where the contraction is large enough.
//
// Both contractions (logits X B, gradient X^T R) are the same kernel: D[128 x N]
// = sum over K of A[128 x K] B[N x K]^T with A a tile of X (rows as M and
// features as K in pass A, features as M and rows as K in pass B).  FP32
// operands are split into three BF16 terms each, h + m + l == x: h is x rounded to six
// significant bits, m the rest rounded to eight, l what is left (exact).  Eight of the
// nine products are formed; ll lies below 2^-30 of |a b|.
//
// Precision.  An MMA aligns its 16 products (and the accumulator) at 2^-25 of the largest,
// cuts off what lies below, adds exactly and truncates the sum to FP32: a sum that does not
// fit loses half its last bit on average, always towards zero, and a chain of MMAs into one
// accumulator shrinks by 1.2e-8 an MMA (X and coefficients ~ N(0, 1), eight-bit h).  Means
// over rows, as log K, and sums over rows, as the gradient, keep such a drift.  So an
// accumulator takes one MMA of hh only, whose 12-bit products add without a truncation
// but for rare spreads, the seven small products of a step of 64 have one of their own
// (2^-7 of the sum, of either sign), and the drain warps add them all to running sums in
// registers with compensated FP32 additions (Kahan).  Bias and spread of a dot product of
// 768 values, relative to the spread of the sums, by a model of that arithmetic which
// reproduces the measured drift: X ~ N(0, 1) -2e-9 and 3e-8 (FMA chains on CUDA cores, 24 a lane:
// 1e-9 and 1.1e-7), pixels -3e-10 and 3e-8 (1e-10 and 8e-8), all positive -1e-9 and 6e-9 (0 and
// 4e-8).  With eight-bit h and six products the bias is -1.2e-8, and -9e-8 with 128
// values of K to an accumulator.  Measured, error of the gradient and of log K against 64
// bits, CUDA cores -> here: normal n=1e4 p=5000 K=10 2.6e-7 -> 8e-8 and 9e-10 -> 5e-10,
// n=5e4 p=1e4 K=20 5.0e-7 -> 8e-8 and 2e-9 -> 6e-10; pixels n=6e4 p=785 K=10 5.1e-8 -> 5.1e-8
// and 1e-9 -> 1e-9; 0/1 indicators there 5.6e-8 -> 4.9e-8 and 1e-9 -> 9e-10.  (Eight-bit h,
// 128 of K to an accumulator, half of a mean drift given back: pixels 6.9e-8 and 3e-8,
// normal 1.8e-7 and 2.7e-8.)  X = exp(1.5 N(0, 1)), whose products spread widest, keeps a
// drift of 7e-9 in log K; its gradients are no further off than the CUDA cores'.
// What it costs, us a gradient, with that form and so: n=1e4 p=5000 K=10 83 -> 90,
// n=6e4 p=785 86 -> 93, n=1e4 p=2e4 K=20 272 -> 300, more than 32 columns n=2e4 p=1000,
// 72 columns in two launches, 78 -> 145, n=5e4 p=1e4, 76 columns, 830 -> 1960: 32 MMAs a
// step for 20, and five accumulators to drain every 64 of K for two every 128.
//
// Why TMEM for A.  Splitting writes 6 bytes for each 4 read, and every MMA reads
// its A operand again: through shared memory this traffic alone (TMA write, split
// read, split write, MMA reads) would take as long as HBM takes to deliver X.
// With A in TMEM, shared memory sees X once in and once out.
//
// X layout: boxes of 64 rows x 64 features, 16 KB, [row block][feature block];
// in a box 16-byte chunk j (features 4j .. 4j + 3) of row r lies at
// j * 1024 + ((r ^ j) & 63) * 16.  A thread of pass A reads its row's chunks with
// 16-byte loads, a thread of pass B its feature's values of 64 rows with 4-byte
// loads; both are free of bank conflicts, and every box is one contiguous copy.
//
// Roles (20 warps): 0 and 1 producers (bulk copies of X and of B), 2 and 3 MMA issuers, 4-7
// and 8-11 converters (two groups that take alternate K steps, each with an A buffer),
// 12-19 drain warps (two per TMEM lane quarter).  Each issuer has a set of accumulators:
// with up to 32 columns the issuers take alternate K steps, with more (kB = 4) the first
// 32 columns and the rest of every step, so that X is split once for all of them; one's
// waits (about 250 clocks each) and drains pass while the other's MMAs run.
// Work: the (tile, K step) pairs are split evenly over the CTAs; a tile that spans
// several CTAs leaves one partial per CTA, summed in CTA order by the next kernel
// (bitwise repeatable, no atomics).
//
// Every wait is bounded; a wait that runs out sets an error bit and an abort
// flag, and every role leaves its loop.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "tc_common.cuh"

namespace hmc {
namespace split {

using tc::fence_after_sync;
using tc::fence_before_sync;
using tc::idesc_bf16;
using tc::mma_commit;
using tc::smem_desc;
using tc::tmem_alloc;
using tc::tmem_dealloc;

constexpr int kBlk = 64;                     // rows and features of a box
constexpr int kBoxBytes = kBlk * kBlk * 4;   // 16 KB
constexpr int64_t kKeepBytes = int64_t(32) << 20;   // of X, see the producer
constexpr int kXSlot = 2 * kBoxBytes;        // one 128 x 64 (or 64 x 128) step of X
constexpr int kThreads = 20 * 32;
constexpr int kACols = 96;                   // TMEM columns of one A buffer: 3 terms x 32 words
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxN = kSplitMaxN;
constexpr int kHalfN = 32;                   // columns of a set of accumulators at most: five each, 2 A buffers + 2 sets = 512

// D[tmem] (+)= A[tmem] B[smem], BF16 operands, FP32 accumulation.
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Eight or four columns of an accumulator (no wait; tmem_ld_wait orders the reads).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
// Two FP32 additions, rounded to nearest, in one instruction.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(*reinterpret_cast<uint64_t*>(&a)), "l"(*reinterpret_cast<uint64_t*>(&b)));
  return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Exact split of a pair of finite FP32 values into BF16 terms, packed with x0 in the low
// half: h rounded to six significant bits (on the upper halves of both values at once:
// bit 17 of an FP32 number is half the last bit kept; an h that would overflow stays at
// the largest finite one), m what remains rounded to eight, l the rest.  The
// subtractions are exact.
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = (__byte_perm(__float_as_uint(x0), __float_as_uint(x1), 0x7632) + 0x00020002u) & 0xfffcfffcu;
  asm("min.xorsign.abs.bf16x2 %0, %0, %1;" : "+r"(h) : "r"(0x7f7c7f7cu));
  const float r0 = x0 - __uint_as_float(h << 16), r1 = x1 - __uint_as_float(h & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(r1), "f"(r0));
  const float s0 = r0 - __uint_as_float(m << 16), s1 = r1 - __uint_as_float(m & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(s1), "f"(s0));
}

// The B side, one value.  An infinite or NaN one stays in h alone (what it makes of the
// small products is left out of the sum, see the drain).  Selects, no branches: with an
// early return for these the softmax of n=6e4, 9 columns took 11.1 us for 7.8.
__device__ __forceinline__ void split_one(float v, uint16_t& h, uint16_t& m, uint16_t& l) {
  const uint32_t u = __float_as_uint(v);
  const bool odd = (u & 0x7f800000u) == 0x7f800000u;
  uint32_t t = (u + 0x20000u) & 0xfffc0000u;
  t = (t & 0x7f800000u) == 0x7f800000u ? (u & 0x80000000u) | 0x7f7c0000u : t;   // would round to infinity
  t = odd ? u | (v != v ? 0x400000u : 0u) : t;
  h = uint16_t(t >> 16);
  const float r = odd ? 0.f : v - __uint_as_float(t);
  const __nv_bfloat16 mb = __float2bfloat16_rn(r);
  m = __bfloat16_as_ushort(mb);
  l = __bfloat16_as_ushort(__float2bfloat16_rn(r - __bfloat162float(mb)));
}

__host__ __device__ inline size_t al(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Args {
  const unsigned char* xs;   // X boxes [nrb][nfb][16 KB]
  const unsigned char* bs;   // B operand [group][halves of K steps][3N rows x 64 B], 64-byte swizzle
  float* out;                // pass A: partial logits [slot][unit][N][128]; pass B: gradient slices [slot][C][p_pad]
  int64_t out_stride;        // elements between slots
  int* err;
  int64_t nrb, nfb;          // row and feature blocks of X
  int64_t ntiles;            // tiles of 128 along M
  int32_t groups;            // column groups (units (group, tile); group g's boxes follow group g - 1's)
  int32_t ksteps;            // steps of 64 along K
  int32_t N, C, p_pad, nslots;
  int32_t nstx, nstb;        // ring slots, half of each ring: X steps, halves of B steps
  int64_t keep_rb;           // row blocks of X kept in L2 (the rest is streamed through it)
  long long spin_limit;
};

struct Smem {
  size_t xring, bring, bars, total;
};
__host__ __device__ inline Smem smem_layout(int nstx, int nstb, int N) {
  Smem L;
  size_t off = 0;
  L.xring = off;  off += size_t(2 * nstx) * kXSlot;
  L.bring = off;  off = al(off + size_t(2 * nstb) * 3 * N * 64, 1024);
  // xfull, xempty [2 nstx]; bfull, bempty [2 nstb]; afull, afree [4]; dfull, dfree, mdrain [2]; TMEM slot; abort flag
  L.bars = off;   off = al(off + size_t(4 * nstx + 4 * nstb + 14 + 2) * 8, 16);
  L.total = off + 1024;   // slack for aligning the dynamic base to 1024
  return L;
}

// One stretch of a CTA's steps: tile group u, K steps [k0, k1).
struct Seg {
  int u;       // unit: tile, or (group, tile) with the tile fastest
  int k0, k1;
};
__device__ __forceinline__ bool next_seg(int& pos, int end, int ksteps, Seg& sg) {   // a launch has fewer than 2^31 steps
  if (pos >= end) return false;
  sg.u = pos / ksteps;
  sg.k0 = pos - sg.u * ksteps;
  sg.k1 = min(ksteps, sg.k0 + (end - pos));
  pos += sg.k1 - sg.k0;
  return true;
}
// The CTA (of G, sharing W steps evenly) that holds step s.
__host__ __device__ inline int64_t cta_of_step(int64_t s, int64_t W, int64_t G) { return ((s + 1) * G - 1) / W; }

// kGrad: false pass A (tile = 128 rows, K = features), true pass B (tile = 128 features, K = rows).
// kB: N <= 16 kB; 2: the issuers take alternate steps, 4: halves of the columns.
template <bool kGrad, int kB>
__global__ void __launch_bounds__(kThreads, 1) gemm_kernel(const Args A) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr bool kHalves = kB > 2;
  const int N = A.N, NX = A.nstx, NB = A.nstb;        // ring slots
  const Smem Lo = smem_layout(NX, NB, N);
  unsigned char* xring = smem + Lo.xring;
  unsigned char* bring = smem + Lo.bring;
  uint64_t* xfull = reinterpret_cast<uint64_t*>(smem + Lo.bars);
  uint64_t* xempty = xfull + 2 * NX;   // xfull, xempty [2 converter groups][NX]
  uint64_t* bfull = xempty + 2 * NX;   // bfull, bempty [2 issuers][NB], or [2 NB] for both
  uint64_t* bempty = bfull + 2 * NB;
  uint64_t* afull = bempty + 2 * NB; // [2 buffers][2 halves] half an A buffer (32 of K) is converted
  uint64_t* afree = afull + 4;       // [2][2] the MMAs reading it are complete
  uint64_t* dfull = afree + 4;       // [2] a step's sums are in the issuer's accumulators
  uint64_t* dfree = dfull + 2;       // [2] drained
  uint64_t* mdrain = dfree + 2;      // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mdrain + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(mdrain + 3);

  if (tid == 0) {
    for (int s = 0; s < 2 * NX; ++s) {
      mbar_init(&xfull[s], 1);
      mbar_init(&xempty[s], 4);
    }
    for (int s = 0; s < 2 * NB; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], kHalves ? 2 : 1);
    }
    for (int a = 0; a < 4; ++a) {
      mbar_init(&afull[a], 4);
      mbar_init(&afree[a], kHalves ? 2 : 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&dfull[a], 1);
      mbar_init(&dfree[a], 8);
      mbar_init(&mdrain[a], 1);
    }
    *abort_flag = 0;
    fence_mbar_init_cluster();
  }
  if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = __reduce_or_sync(0xffffffffu, *tmem_slot);

  const int64_t W = A.groups * A.ntiles * A.ksteps, G = gridDim.x;
  const int s_end = int((int64_t(blockIdx.x) + 1) * W / G);
  const uint32_t bbytes = uint32_t(3 * N * 64);
  auto fail = [&](int bit) {
    *abort_flag = 1;
    atomicOr(A.err, bit);
  };
  // The whole warp waits, for up to three barriers at once, and agrees on the outcome.
  // Every branch on an issuing warp's path costs some 25 clocks, so the probes are
  // combined before the one branch of the fast path.
  const bool live = A.spin_limit > 0;   // fault injection: every wait gives up at once
  auto wait_warp3 = [&](uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, uint64_t* b2, uint32_t p2, int bit) {
    const uint32_t a0 = smem_u32(b0), a1 = smem_u32(b1), a2 = smem_u32(b2);
    auto probe = [&]() {
      bool r = mbar_test_cta(a0, p0) & live;
      if (b1 != b0) r &= mbar_test_cta(a1, p1);      // the same barrier twice: decided at compile time
      if (b2 != b0) r &= mbar_test_cta(a2, p2);
      return bool(__all_sync(0xffffffffu, r));
    };
    if (probe()) return true;
    for (long long i = 1; i < A.spin_limit; ++i) {
      if (probe()) return true;
      if ((i & 63) == 63 && __any_sync(0xffffffffu, *abort_flag != 0)) break;
    }
    if (lane == 0) fail(bit);
    return false;
  };
  auto wait_warp2 = [&](uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, int bit) {
    return wait_warp3(b0, p0, b1, p1, b0, p0, bit);
  };
  auto wait_warp = [&](uint64_t* bar, uint32_t parity, int bit) {
    return wait_warp3(bar, parity, bar, parity, bar, parity, bit);
  };
  int pos = int(int64_t(blockIdx.x) * W / G);
  Seg sg;

  if (warp < 2) {
    // ------------------------------------------------------------ producers (0: X, 1: B)
    // Converter groups and issuers that take alternate steps have rings of their own; issuers
    // that take every step both free a slot of the one ring.  So a consumer meets all uses of
    // a slot, and no wait can be a full round ahead of the barrier's phase.
    const int n = warp == 0 ? NX : kHalves ? 2 * NB : NB;
    uint64_t* full = warp == 0 ? xfull : bfull;
    uint64_t* empty = warp == 0 ? xempty : bempty;
    Ring r0, r1;
    int uses0 = 0, uses1 = 0;            // up to n: the uses that may be in flight at the end
    uint32_t s = 0;
    bool ok = true;
    // X larger than L2 would push out the B operand, the residuals and the partials:
    // it is streamed with evict-first priority, but for its first rows, which the next
    // pass finds again (n=1e4 p=5000 K=10, when a pass took 37 us for the 41 of now: 80.5 us a
    // leapfrog step with no priorities, 75.9 all evict-first, 75.4 with 30 MB kept, 77.9
    // with 70 MB; from a cold L2 107, 104 and 97 us a gradient; four handles in turn 89.6
    // all evict-first, 92.2 with 32 MB of each kept).
    const uint64_t keep = l2_evict_last(), stream = l2_evict_first();
    // X is what no kernel of the chain writes: its first copies need not wait for the
    // kernel before this one.
    if (warp == 1) chain_wait();
    auto slot_wait = [&](Ring& r, int& uses, int line) {
      ok = wait_warp(&empty[line * n + r.slot], r.par ^ 1u, ERR_TIMEOUT_STAGE);
      if (ok && uses < n) ++uses;
      return ok;
    };
    while (ok && next_seg(pos, s_end, A.ksteps, sg)) {
      const int64_t g = sg.u / A.ntiles, t = sg.u - g * A.ntiles;
      const unsigned char* bg = A.bs + size_t(g) * A.ksteps * 2 * bbytes;
      for (int k = sg.k0; k < sg.k1 && ok; ++k, ++s) {
        const int line = (warp == 0 || !kHalves) ? int(s & 1u) : 0;
        Ring& r = line ? r1 : r0;
        int& uses = line ? uses1 : uses0;
        if (warp == 1) {
          for (int hb = 0; hb < 2; ++hb) {
            if (!slot_wait(r, uses, line)) break;
            if (tc::elect_one()) {
              uint64_t* bar = &full[line * n + r.slot];
              mbar_arrive_expect_tx(bar, bbytes);
              bulk_g2s(bring + uint32_t(line * n + r.slot) * bbytes, bg + size_t(2 * k + hb) * bbytes, bbytes, bar);
            }
            __syncwarp();
            r.next(n);
          }
        } else {
          if (!slot_wait(r, uses, line)) break;
          if (tc::elect_one()) {
            uint64_t* bar = &full[line * n + r.slot];
            unsigned char* dst = xring + uint32_t(line * n + r.slot) * uint32_t(kXSlot);
            if (kGrad) {
              // feature blocks 2t, 2t + 1 of row block k are neighbours
              const uint32_t by = 2 * t + 1 < A.nfb ? uint32_t(kXSlot) : uint32_t(kBoxBytes);
              mbar_arrive_expect_tx(bar, by);
              bulk_g2s_hint(dst, A.xs + size_t(k * A.nfb + 2 * t) * kBoxBytes, by, bar, k < A.keep_rb ? keep : stream);
            } else {
              const bool two = 2 * t + 1 < A.nrb;
              mbar_arrive_expect_tx(bar, two ? uint32_t(kXSlot) : uint32_t(kBoxBytes));
              const uint64_t pol = 2 * t < A.keep_rb ? keep : stream;
              bulk_g2s_hint(dst, A.xs + size_t(2 * t * A.nfb + k) * kBoxBytes, kBoxBytes, bar, pol);
              if (two)
                bulk_g2s_hint(dst + kBoxBytes, A.xs + size_t((2 * t + 1) * A.nfb + k) * kBoxBytes, kBoxBytes, bar, pol);
            }
          }
          __syncwarp();
          r.next(n);
        }
      }
    }
    // Every copy issued must land before shared memory is released: walk back over
    // the last uses of both rings.
    for (int line = 0; line < 2; ++line) {
      Ring& r = line ? r1 : r0;
      for (int q = line ? uses1 : uses0; q > 0; --q) {
        if (r.slot == 0) {
          r.slot = n;
          r.par ^= 1u;
        }
        --r.slot;
        wait_drain(&full[line * n + r.slot], r.par, A.spin_limit);
      }
    }
  } else if (warp < 4) {
    // ------------------------------------------------------------ MMA issuers
    // The whole warp runs the loop, one elected lane issues.  A step: per half (32 of K)
    // two MMAs of hh, each into an accumulator of its own, and fourteen of the small
    // products into the set's fifth accumulator.
    const int g = warp - 2;
    const int Ng = !kHalves ? N : g == 0 ? kHalfN : N - kHalfN, c0 = kHalves ? g * kHalfN : 0;   // columns, the first
    const uint32_t id = idesc_bf16(128, Ng, false, false);
    const uint32_t d0 = tmem + uint32_t(2 * kACols + g * 5 * (kHalves ? kHalfN : N)), d1 = d0 + uint32_t(4 * Ng);
    const uint32_t b0 = smem_u32(bring) + uint32_t(c0 * 64);
    const uint64_t desc_hi = smem_desc(0u, 16u, 512u, 4u);
    const uint64_t nterm = uint64_t(N) * 4;            // one term of the B box, in descriptor units
    const int ring0 = kHalves ? 0 : g * NB, nring = kHalves ? 2 * NB : NB;
    uint32_t s0 = 0;                                   // steps of the CTA before this segment
    Ring br;
    bool ok = true;
    while (ok && next_seg(pos, s_end, A.ksteps, sg)) {
      const int cnt = sg.k1 - sg.k0;
      for (int c = kHalves ? 0 : int(s0 & 1u) ^ g; c < cnt; c += kHalves ? 1 : 2) {
        const uint32_t s = s0 + uint32_t(c), ab = s & 1u, apar = (s >> 1) & 1u;
        const uint32_t epar = (kHalves ? ab : apar) ^ 1u;       // dfree's phase of this issuer's step before
        const uint32_t abuf = kHalves ? tc::uniform(tmem + ab * uint32_t(kACols)) : tmem + uint32_t(g * kACols);
#pragma unroll
        for (int hb = 0; hb < 2; ++hb) {
          const int slot = ring0 + br.slot;
          // The first half also waits for the accumulators.
          ok = hb == 0 ? wait_warp3(&afull[2 * ab], apar, &bfull[slot], br.par, &dfree[g], epar, ERR_TIMEOUT_STAGE)
                       : wait_warp2(&afull[2 * ab + 1], apar, &bfull[slot], br.par, ERR_TIMEOUT_STAGE);
          if (!ok) break;
          fence_after_sync();
          // The reduction puts the warp-uniform address into a uniform register, where
          // the MMAs take their descriptors from.
          const uint64_t dh0 = desc_hi | __reduce_or_sync(0xffffffffu, (b0 + uint32_t(slot) * bbytes) >> 4);
          if (tc::elect_one()) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const uint64_t dh = dh0 + uint64_t(2 * q), dm = dh + nterm, dl = dm + nterm;
              const uint32_t xh = abuf + uint32_t(hb * 48 + 8 * q), xm = xh + 16u, xl = xh + 32u;
              mma_ts(d0 + uint32_t((2 * hb + q) * Ng), xh, dh, id, 0u);   // hh
              mma_ts(d1, xh, dm, id, (hb > 0 || q > 0) ? 1u : 0u);        // hm
              mma_ts(d1, xm, dh, id, 1u);                                 // mh
              mma_ts(d1, xm, dm, id, 1u);                                 // mm
              mma_ts(d1, xh, dl, id, 1u);                                 // hl
              mma_ts(d1, xl, dh, id, 1u);                                 // lh
              mma_ts(d1, xm, dl, id, 1u);                                 // ml
              mma_ts(d1, xl, dm, id, 1u);                                 // lm
            }
            mma_commit(&afree[2 * ab + hb]);
            mma_commit(&bempty[slot]);
            if (hb == 1) mma_commit(&dfull[g]);
          }
          __syncwarp();
          br.next(nring);
        }
        if (!ok) break;
      }
      s0 += uint32_t(cnt);
    }
    // TMEM and shared memory stay allocated until every MMA has completed.
    if (tc::elect_one()) mma_commit(&mdrain[g]);
    __syncwarp();
    wait_drain(&mdrain[g], 0u, A.spin_limit);
  } else if (warp < 12) {
    // ------------------------------------------------------------ converters, two groups of four warps
    const int g = (warp - 4) >> 2;
    const int q = warp & 3;                          // TMEM lane quarter
    const uint32_t ta = tmem + uint32_t(g * kACols) + (uint32_t(32 * q) << 16);
    const int in_blk = 32 * (q & 1) + lane;          // row (pass A) or feature (pass B) within its box
    const unsigned char* xq = xring + (q >> 1) * kBoxBytes;
    uint32_t s0 = 0, mine = 0;                       // steps of the CTA before this segment, of this group so far
    Ring xr;
    bool ok = true;
    while (ok && next_seg(pos, s_end, A.ksteps, sg)) {
      const int cnt = sg.k1 - sg.k0;
      for (int c = int(s0 & 1u) ^ g; c < cnt; c += 2, xr.next(NX)) {
        const uint32_t apar = (mine & 1u) ^ 1u;        // afree's phase of this group's step before
        const unsigned char* xb = xq + uint32_t(g * NX + xr.slot) * uint32_t(kXSlot);
#pragma unroll
        for (int hb = 0; hb < 2; ++hb) {
          ok = hb == 0 ? wait_warp2(&afree[2 * g], apar, &xfull[g * NX + xr.slot], xr.par, ERR_TIMEOUT_STAGE)
                       : wait_warp(&afree[2 * g + 1], apar, ERR_TIMEOUT_STAGE);
          if (!ok) break;
          fence_after_sync();
          const uint32_t th = ta + uint32_t(48 * hb);  // h, m, l: 16 columns each
#pragma unroll
          for (int b = 0; b < 2; ++b) {                // 16 of K: 8 words of each term
            uint32_t h[8], m[8], l[8];
            if (!kGrad) {
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) {
                const int j = 8 * hb + 4 * b + jj;
                const float4 v = *reinterpret_cast<const float4*>(xb + j * 1024 + ((in_blk ^ j) << 4));
                split_pair(v.x, v.y, h[2 * jj], m[2 * jj], l[2 * jj]);
                split_pair(v.z, v.w, h[2 * jj + 1], m[2 * jj + 1], l[2 * jj + 1]);
              }
            } else {
              const int j = in_blk >> 2;
              const unsigned char* xe = xb + j * 1024 + (in_blk & 3) * 4 + (2 * hb + b) * 256;
#pragma unroll
              for (int rr = 0; rr < 8; ++rr) {
                const float x0 = *reinterpret_cast<const float*>(xe + (((2 * rr) ^ j) << 4));
                const float x1 = *reinterpret_cast<const float*>(xe + (((2 * rr + 1) ^ j) << 4));
                split_pair(x0, x1, h[rr], m[rr], l[rr]);
              }
            }
            tmem_st8(th + 8u * b, h);
            tmem_st8(th + 16u + 8u * b, m);
            tmem_st8(th + 32u + 8u * b, l);
          }
          tmem_st_wait();
          fence_before_sync();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive_local(&afull[2 * g + hb]);
            if (hb == 1) mbar_arrive_local(&xempty[g * NX + xr.slot]);
          }
        }
        if (!ok) break;
        ++mine;
      }
      s0 += uint32_t(cnt);
    }
  } else {
    // ------------------------------------------------------------ drain
    // Running sums in FP32 with the rounding errors carried along (Kahan): x is added to
    // acc + cmp.  An infinite sum stays what it is: its correction (NaN) becomes a finite
    // number, and so do the small products, NaN where a coefficient is infinite.
    const int q = warp & 3, hf = (warp - 12) >> 2;   // lane quarter; blocks of 8 columns of a set: hf, hf + 2
    const int mrow = 32 * q + lane;
    const uint32_t tq = tmem + uint32_t(2 * kACols + 8 * hf) + (uint32_t(32 * q) << 16);
    constexpr int kSets = kHalves ? 2 : 1;           // of a step
    float2 acc[kSets][2][4], cmp[kSets][2][4];
    chain_wait();                                    // the sums' buffer may still be read
    uint32_t s = 0;
    bool ok = true;
    while (ok && next_seg(pos, s_end, A.ksteps, sg)) {
#pragma unroll
      for (int h = 0; h < kSets; ++h)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[h][b][e] = cmp[h][b][e] = make_float2(0.f, 0.f);
      for (int k = sg.k0; k < sg.k1 && ok; ++k, ++s) {
#pragma unroll
        for (int h = 0; h < kSets; ++h) {
          const uint32_t a = kHalves ? uint32_t(h) : s & 1u, par = (kHalves ? s : s >> 1) & 1u;
          const int Ng = !kHalves ? N : h == 0 ? kHalfN : N - kHalfN;
          const uint32_t t0 = tq + a * uint32_t(5 * (kHalves ? kHalfN : N));
          if (!(ok = wait_warp(&dfull[a], par, ERR_TIMEOUT_MMA))) break;
          fence_after_sync();
          constexpr int kW = kHalves ? 4 : 8;        // columns at a time (registers)
#pragma unroll
          for (int b = 0; b < 2; ++b)
            if (16 * b + 8 * hf < Ng) {
#pragma unroll
              for (int e0 = 0; e0 < 8; e0 += kW) {
                uint32_t v[5][kW];
#pragma unroll
                for (int i = 0; i < 5; ++i)
                  if constexpr (kW == 8) tmem_ld8(t0 + uint32_t(i * Ng + 16 * b), v[i]);
                  else tmem_ld4(t0 + uint32_t(i * Ng + 16 * b + e0), v[i]);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < kW; e += 2) {
                  auto f = [&](int i) { return make_float2(__uint_as_float(v[i][e]), __uint_as_float(v[i][e + 1])); };
                  const float2 lo = make_float2(fmaxf(fminf(f(4).x, 3e38f), -3e38f), fmaxf(fminf(f(4).y, 3e38f), -3e38f));
                  const float2 x = add2(add2(add2(f(0), f(1)), add2(f(2), f(3))), lo);
                  float2 &sum = acc[h][b][(e0 + e) / 2], &err = cmp[h][b][(e0 + e) / 2];
                  const float2 y = add2(x, err), t = add2(sum, y);
                  err = add2(y, neg2(add2(t, neg2(sum))));
                  err = make_float2(fminf(err.x, 1e30f), fminf(err.y, 1e30f));
                  sum = t;
                }
              }
            }
          fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive_local(&dfree[a]);
        }
      }
      if (!ok) break;
      // This CTA's partial of the tile: its place among the tile's CTAs.
      const int64_t t = sg.u;   // pass B has one group: the unit is the tile
      const int64_t sl = int64_t(blockIdx.x) - cta_of_step(t * A.ksteps, W, G);
      float* out = A.out + size_t(sl) * A.out_stride;
#pragma unroll
      for (int h = 0; h < kSets; ++h)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int c = h * kHalfN + 16 * b + 8 * hf + e;
            const float2 sum = add2(acc[h][b][e / 2], cmp[h][b][e / 2]);
            if (c >= A.C) continue;
            if (kGrad) {
              const int64_t col = t * 128 + mrow;
              if (col < A.p_pad) {
                out[size_t(c) * A.p_pad + col] = e & 1 ? sum.y : sum.x;
                // The tile's last CTA clears the slots that no CTA fills.
                if (sg.k1 == A.ksteps)
                  for (int64_t z = sl + 1; z < A.nslots; ++z)
                    A.out[size_t(z) * A.out_stride + size_t(c) * A.p_pad + col] = 0.f;
              }
            } else {
              out[(size_t(t) * N + c) * 128 + mrow] = e & 1 ? sum.y : sum.x;
            }
          }
    }
    fence_before_sync();
  }
  __syncthreads();
  if (warp == 0) {
    fence_after_sync();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// Coefficients [C][p_pad] -> operand boxes [p_pad / 32][3N rows x 64 B] (h, m, l
// rows of each column; 64-byte swizzle: chunk ^ (row / 2) % 4).  One thread: 8 consecutive features of a
// column, one 16-byte chunk of each term.  Columns past C are left as they are:
// they only reach accumulator columns nobody reads.
__global__ void coef_boxes_kernel(const float* __restrict__ beta, unsigned char* __restrict__ out, int32_t C, int32_t N,
                                  int32_t p_pad) {
  chain_wait();
  chain_next();
  const int p8 = p_pad / 8;
  const int64_t total = int64_t(C) * p8;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int c = int(i / p8);
    const int col = 8 * int(i - int64_t(c) * p8);
    const float4 a = *reinterpret_cast<const float4*>(beta + size_t(c) * p_pad + col);
    const float4 b = *reinterpret_cast<const float4*>(beta + size_t(c) * p_pad + col + 4);
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t w[3][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint16_t t0[3], t1[3];
      split_one(v[2 * k], t0[0], t0[1], t0[2]);
      split_one(v[2 * k + 1], t1[0], t1[1], t1[2]);
#pragma unroll
      for (int t = 0; t < 3; ++t) w[t][k] = uint32_t(t0[t]) | uint32_t(t1[t]) << 16;
    }
    unsigned char* box = out + size_t(col / 32) * 3 * N * 64;
    const int chunk = ((col % 32) >> 3) ^ ((c >> 1) & 3);   // N is a multiple of 8: the terms' rows share the swizzle
#pragma unroll
    for (int t = 0; t < 3; ++t)
      *reinterpret_cast<uint4*>(box + size_t(t * N + c) * 64 + (chunk << 4)) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
  }
}

// Softmax of one 64-row block (Eqs. softmax, loglike): sums the partial logits of
// the CTAs that share the rows' tile in CTA order, forms every chain's
// log-likelihood (FP64 sum over the block's rows in a fixed tree) and writes the
// residual Y - P as the split operand boxes of pass B (zero on rows past n).
// Bound by latency: loads, one chain of exponentials per (row, chain), stores; a
// thread writes eight rows of a column as one 16-byte chunk of each term.
constexpr int kSoftThreads = 256;
constexpr int kSoftPitch = kBlk + 4;   // floats of a column in shared memory (16-byte chunks of 8 columns spread over the banks)
__global__ void __launch_bounds__(kSoftThreads) softmax_kernel(const float* __restrict__ zpart, int64_t slot_stride,
                                                              const int32_t* __restrict__ y,
                                                              unsigned char* __restrict__ rb, double* __restrict__ lblk,
                                                              int32_t lstride, int64_t n, int32_t C, int32_t N,
                                                              int32_t Km1, int32_t chains, int32_t zlogit,
                                                              int64_t ksteps, int64_t W, int64_t G, int* err) {
  extern __shared__ __align__(16) float zs[];          // [C] logits, then exponentials; [chains] 1 / normaliser
  float* is = zs + size_t(C) * kSoftPitch;
  double* ls = reinterpret_cast<double*>(is + size_t(chains) * kSoftPitch);   // [chains][2]: half sums
  int* ys = reinterpret_cast<int*>(ls + 2 * size_t(chains));                  // [64]
  chain_wait();
  chain_next();
  const int r = threadIdx.x & (kBlk - 1), tg = threadIdx.x >> 6;              // row, column group (of 4)
  const int64_t blk = blockIdx.x, row = blk * kBlk + r;
  const int64_t tile = blk >> 1;
  const int nsl = int(cta_of_step((tile + 1) * ksteps - 1, W, G) - cta_of_step(tile * ksteps, W, G)) + 1;
  const int mrow = int(blk & 1) * kBlk + r;
  const bool valid = row < n;
  int yi = valid ? __ldg(y + row) : 0;
  if (yi < 0 || yi >= Km1 + zlogit) {
    atomicOr(err, ERR_BAD_LABEL);
    yi = 0;
  }
  if (tg == 0) ys[r] = yi;
  {
    const float* z = zpart + size_t(tile) * N * 128 + mrow;
    int c = tg;
    for (; c + 12 < C; c += 16) {                       // four columns in flight
      float v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = valid ? z[size_t(c + 4 * i) * 128] : 0.f;
      for (int s = 1; s < nsl; ++s)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] += valid ? z[size_t(s) * slot_stride + size_t(c + 4 * i) * 128] : 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) zs[(c + 4 * i) * kSoftPitch + r] = v[i];
    }
    for (; c < C; c += 4) {
      float v = valid ? z[size_t(c) * 128] : 0.f;
      for (int s = 1; s < nsl; ++s) v += valid ? z[size_t(s) * slot_stride + size_t(c) * 128] : 0.f;
      zs[c * kSoftPitch + r] = v;
    }
  }
  __syncthreads();
  for (int ch = tg; ch < chains; ch += kSoftThreads / kBlk) {
    float* z = zs + size_t(ch) * Km1 * kSoftPitch + r;
    float m = zlogit ? 0.f : -INFINITY;
    for (int k = 0; k < Km1; ++k) m = fmaxf(m, z[k * kSoftPitch]);
    const float zy = yi < Km1 ? z[yi * kSoftPitch] : 0.f;   // yi == Km1: class K, logit 0
    float sum = zlogit ? expf(-m) : 0.f;
    for (int k = 0; k < Km1; ++k) {
      const float e = expf(z[k * kSoftPitch] - m);
      z[k * kSoftPitch] = e;
      sum += e;
    }
    is[ch * kSoftPitch + r] = 1.f / sum;
    double ll = valid ? double(zy - m - logf(sum)) : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ll += __shfl_xor_sync(0xffffffffu, ll, o);   // 32 rows of one warp
    if ((r & 31) == 0) ls[ch * 2 + (r >> 5)] = ll;
  }
  __syncthreads();
  if (int(threadIdx.x) < chains)
    lblk[size_t(blk) * lstride + threadIdx.x] = ls[threadIdx.x * 2] + ls[threadIdx.x * 2 + 1];
  const int rows = int(min(int64_t(kBlk), n - blk * kBlk));
  for (int t = threadIdx.x; t < 8 * C; t += kSoftThreads) {
    const int c = t >> 3, r8 = (t & 7) * 8, ch = c / Km1, k = c - ch * Km1;
    const float* e = zs + c * kSoftPitch + r8;
    const float* iv = is + ch * kSoftPitch + r8;
    uint32_t w[3][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint16_t a[3], b[3];
      const int r0 = r8 + 2 * q;
      split_one(r0 < rows ? (ys[r0] == k ? 1.f : 0.f) - e[2 * q] * iv[2 * q] : 0.f, a[0], a[1], a[2]);
      split_one(r0 + 1 < rows ? (ys[r0 + 1] == k ? 1.f : 0.f) - e[2 * q + 1] * iv[2 * q + 1] : 0.f, b[0], b[1], b[2]);
#pragma unroll
      for (int j = 0; j < 3; ++j) w[j][q] = uint32_t(a[j]) | uint32_t(b[j]) << 16;
    }
    unsigned char* d = rb + size_t(2 * blk + (r8 >> 5)) * 3 * N * 64 + size_t(c) * 64 +
                       ((((r8 & 31) >> 3) ^ ((c >> 1) & 3)) << 4);
#pragma unroll
    for (int j = 0; j < 3; ++j)
      *reinterpret_cast<uint4*>(d + size_t(j) * N * 64) = make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
  }
}

// ------------------------------------------------------- posterior predictive
// Coefficient draws [ndraws][ku][p] -> operand boxes of groups of `dpg` draws
// (columns (draw, class), dpg km1 of them): one thread per 8 features of a column.
// Non-finite values raise *flag.
__global__ void draw_boxes_kernel(const float* __restrict__ draws, unsigned char* __restrict__ out, int64_t ndraws,
                                  int32_t ku, int32_t km1, int32_t p, int32_t p_pad, int32_t dpg, int32_t N, int* flag) {
  const int p8 = p_pad / 8;
  const int64_t total = ndraws * km1 * p8;
  int bad = 0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t dk = i / p8;
    const int col = 8 * int(i - dk * p8);
    const int64_t d = dk / km1;
    const int k = int(dk - d * km1);
    const int64_t g = d / dpg;
    const int c = int(d - g * dpg) * km1 + k;
    const float* src = draws + (size_t(d) * ku + k) * p + col;
    uint32_t w[3][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint16_t t0[3], t1[3];
      const float v0 = col + 2 * q < p ? src[2 * q] : 0.f, v1 = col + 2 * q + 1 < p ? src[2 * q + 1] : 0.f;
      if (!isfinite(v0) || !isfinite(v1)) bad = 1;
      split_one(v0, t0[0], t0[1], t0[2]);
      split_one(v1, t1[0], t1[1], t1[2]);
#pragma unroll
      for (int t = 0; t < 3; ++t) w[t][q] = uint32_t(t0[t]) | uint32_t(t1[t]) << 16;
    }
    unsigned char* box = out + size_t(g * (p_pad / 32) + col / 32) * 3 * N * 64;
    const int chunk = ((col % 32) >> 3) ^ ((c >> 1) & 3);
#pragma unroll
    for (int t = 0; t < 3; ++t)
      *reinterpret_cast<uint4*>(box + size_t(t * N + c) * 64 + (chunk << 4)) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
  }
  if (bad) atomicOr(flag, 1);
}

// Softmax of every (row, draw) of a launch: block (unit, draw of the group), one
// thread per row of the unit's tile.  The partials of the CTAs that share the unit are
// summed in CTA order; the probabilities of the free classes replace the logits of
// slot 0, that of class K (zero logit) goes to pk[draw][row].  Non-finite logits raise
// *flag.  Split from the sums below so that all draws are formed at once: one thread
// per row doing both took 190 of 370 us for 10000 rows and 100 draws, 700 of 800 us
// for 300 rows.
template <int KB>
__global__ void __launch_bounds__(128) predict_prob_kernel(float* __restrict__ zpart, int64_t slot_stride, int64_t ntiles,
                                                          int32_t N, int64_t ksteps, int64_t W, int64_t G, int64_t n,
                                                          int64_t ndraws, int32_t dpg, int32_t km1, int32_t zlogit,
                                                          float* __restrict__ pk, int64_t rows_pad, int* flag) {
  const int64_t u = blockIdx.x / dpg;
  const int j = int(blockIdx.x - u * dpg);
  const int64_t g = u / ntiles, row = (u - g * ntiles) * 128 + threadIdx.x, d = g * dpg + j;
  if (row >= n || d >= ndraws) return;
  const int nsl = int(cta_of_step((u + 1) * ksteps - 1, W, G) - cta_of_step(u * ksteps, W, G)) + 1;
  float* z0 = zpart + (size_t(u) * N + size_t(j) * km1) * 128 + threadIdx.x;
  float z[KB];
#pragma unroll
  for (int k = 0; k < KB; ++k) z[k] = k < km1 ? z0[size_t(k) * 128] : 0.f;
  for (int q = 1; q < nsl; ++q)
#pragma unroll
    for (int k = 0; k < KB; ++k)
      if (k < km1) z[k] += z0[size_t(q) * slot_stride + size_t(k) * 128];
  float m = zlogit ? 0.f : -INFINITY;
  int bad = 0;
#pragma unroll
  for (int k = 0; k < KB; ++k)
    if (k < km1) {
      if (!isfinite(z[k])) bad = 1;
      m = fmaxf(m, z[k]);
    }
  const float e0 = expf(-m);                        // the zero logit of class K
  float t = zlogit ? e0 : 0.f;
#pragma unroll
  for (int k = 0; k < KB; ++k)
    if (k < km1) {
      z[k] = expf(z[k] - m);
      t += z[k];
    }
#pragma unroll
  for (int k = 0; k < KB; ++k)
    if (k < km1) z0[size_t(k) * 128] = z[k] / t;
  if (zlogit) pk[size_t(d) * rows_pad + row] = e0 / t;
  if (bad) atomicOr(flag, 1);
}

// FP64 sums of the probabilities in draw order: block 32 rows x K classes, one thread
// per (row, class), kFlight draws in flight.  Their FP32 probabilities are summed with
// their rounding errors and theirs carried (two-sum, twice; 2^-71 of the sum is dropped)
// before they meet the FP64 sum, which rounds three times where it rounded eight: bound by
// the FP64 units, n=1e4 K=10 and 100 draws took 68 us with a conversion and an addition for
// each, 28 us with the first errors alone, 32 us with both.  `first`: the sums start at zero, else at
// `acc`; total_draws > 0 (last launch): the means and their argmax (lowest class on a
// tie) are written, else the sums go to `acc`.
__global__ void predict_sum_kernel(const float* __restrict__ zpart, int64_t ntiles, int32_t N, int64_t n, int64_t ndraws,
                                   int32_t dpg, int32_t km1, int32_t K, const float* __restrict__ pk, int64_t rows_pad,
                                   double* __restrict__ acc, int first, double total_draws, double* __restrict__ prob,
                                   int32_t* __restrict__ cls) {
  __shared__ double mean[32][33];
  const int lane = threadIdx.x, k = threadIdx.y;
  const int64_t row = int64_t(blockIdx.x) * 32 + lane;
  if (row < n) {
    const int64_t tile = row >> 7;
    const size_t gstep = size_t(ntiles) * N * 128;
    const float* zk = zpart + (size_t(tile) * N + k) * 128 + (row & 127);
    double s = first ? 0.0 : acc[size_t(row) * K + k];
    int64_t g = 0;
    int j = 0;
    constexpr int kFlight = 8;
    for (int64_t d = 0; d < ndraws; d += kFlight) {
      float v[kFlight];
#pragma unroll
      for (int i = 0; i < kFlight; ++i) {
        v[i] = 0.f;
        if (d + i < ndraws) {
          v[i] = k < km1 ? zk[size_t(g) * gstep + size_t(j) * km1 * 128] : pk[size_t(d + i) * rows_pad + row];
          if (++j == dpg) {
            j = 0;
            ++g;
          }
        }
      }
      float hi = v[0], lo = 0.f, rest = 0.f;
#pragma unroll
      for (int i = 1; i < kFlight; ++i) {
        hi = two_sum(hi, v[i], v[i]);
        lo = two_sum(lo, v[i], v[i]);
        rest = __fadd_rn(rest, v[i]);
      }
      s += (double(hi) + double(lo)) + double(rest);
    }
    if (total_draws == 0.0) {
      acc[size_t(row) * K + k] = s;
    } else {
      mean[lane][k] = s / total_draws;
      if (prob) prob[size_t(row) * K + k] = mean[lane][k];
    }
  }
  __syncthreads();
  if (total_draws == 0.0 || !cls || k != 0 || row >= n) return;
  int best = 0;
  for (int q = 1; q < K; ++q)
    if (mean[lane][q] > mean[lane][best]) best = q;
  cls[row] = best;
}

// Rows (IT, n x p) -> X boxes, zero past n and p; flags non-finite values.  One
// block per box, through shared memory so that reads and writes are contiguous.
template <typename IT>
__global__ void __launch_bounds__(256) rows_to_boxes_kernel(const IT* __restrict__ src, float* __restrict__ dst, int64_t n,
                                                            int32_t p, int64_t nfb, int* err) {
  __shared__ float t[kBlk * kBlk];
  const int64_t fb = int64_t(blockIdx.x) % nfb, rbk = int64_t(blockIdx.x) / nfb;
  int bad = 0;
  for (int e = threadIdx.x; e < kBlk * kBlk; e += blockDim.x) {
    const int r = e / kBlk, f = e % kBlk, j = f >> 2;
    const int64_t row = rbk * kBlk + r, col = fb * kBlk + f;
    IT v = IT(0);
    if (row < n && col < p) v = src[row * p + col];
    if (!isfinite(double(v))) bad = 1;
    t[j * 256 + ((r ^ j) << 2) + (f & 3)] = float(v);
  }
  __syncthreads();
  float4* o = reinterpret_cast<float4*>(dst + size_t(blockIdx.x) * kBlk * kBlk);
  for (int e = threadIdx.x; e < kBlk * kBlk / 4; e += blockDim.x) o[e] = reinterpret_cast<const float4*>(t)[e];
  if (bad) atomicOr(err, ERR_NONFINITE_X);
}

// X boxes -> rows (the values as stored).
__global__ void boxes_to_rows_kernel(const float* __restrict__ src, float* __restrict__ dst, int64_t n, int32_t p,
                                     int64_t nfb) {
  const int64_t total = n * p;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t row = i / p, col = i - row * p;
    const int r = int(row % kBlk), f = int(col % kBlk), j = f >> 2;
    dst[i] = src[size_t((row / kBlk) * nfb + col / kBlk) * kBlk * kBlk + j * 256 + ((r ^ j) << 2) + (f & 3)];
  }
}

size_t softmax_smem(int C, int chains) { return size_t(C + chains) * kSoftPitch * 4 + size_t(chains) * 2 * 8 + kBlk * 4; }

}  // namespace split

static void (*split_gemm(bool grad, int N))(const split::Args) {
  if (N <= 32) return grad ? split::gemm_kernel<true, 2> : split::gemm_kernel<false, 2>;
  return grad ? split::gemm_kernel<true, split::kMaxN / 16> : split::gemm_kernel<false, split::kMaxN / 16>;
}

int split_columns(int C) { return std::max(16, (C + 15) / 16 * 16); }

static int64_t split_slots(int64_t groups, int64_t ksteps, int64_t G) {
  const int64_t W = groups * ksteps;
  int64_t m = 1;
  for (int64_t u = 0; u < groups; ++u)
    m = std::max(m, split::cta_of_step((u + 1) * ksteps - 1, W, G) - split::cta_of_step(u * ksteps, W, G) + 1);
  return m;
}

bool split_plan(int64_t n, int64_t p, int C, int nsm, int smem_max, SplitPlan* out) {
  SplitPlan P{};
  if (n < 1 || C < 1 || C > split::kMaxN) return false;
  P.p_pad = int((p + split::kBlk - 1) / split::kBlk * split::kBlk);
  P.nrb = (n + split::kBlk - 1) / split::kBlk;
  P.nfb = P.p_pad / split::kBlk;
  if (P.nrb * P.nfb > int64_t(0x7fffffff)) return false;   // one block per box in the upload, one step per two boxes
  P.N = split_columns(C);
  const int64_t ta = (P.nrb + 1) / 2, tb = (P.nfb + 1) / 2;
  P.gridA = int(std::min<int64_t>(nsm, ta * P.nfb));
  P.gridB = int(std::min<int64_t>(nsm, tb * P.nrb));
  P.slotsA = int(split_slots(ta, P.nfb, P.gridA));
  P.slotsB = int(split_slots(tb, P.nrb, P.gridB));
  // Rings, each half: three halves of a B step, X steps in the rest.
  P.nstb = 3;
  P.nstx = 0;
  for (int s = 3; s >= 2 && !P.nstx; --s)
    if (split::smem_layout(s, P.nstb, P.N).total <= size_t(smem_max)) P.nstx = s;
  if (!P.nstx) return false;
  P.smem = std::max(split::smem_layout(P.nstx, P.nstb, P.N).total, size_t(116 * 1024));   // one CTA per SM
  *out = P;
  return true;
}

cudaError_t split_prepare() {
  int dev = 0, smem_max = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  for (int N : {16, split::kMaxN})
    for (bool grad : {false, true})
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(split_gemm(grad, N), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(split::softmax_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(split::softmax_smem(split::kMaxN, split::kMaxN)));
  return e;
}

size_t split_x_bytes(const SplitPlan& P) { return size_t(P.nrb) * P.nfb * split::kBoxBytes; }
size_t split_box_bytes(const SplitPlan& P, int64_t steps) { return size_t(steps) * 3 * P.N * 128; }
size_t split_zpart_bytes(const SplitPlan& P) {
  return size_t(P.slotsA) * ((P.nrb + 1) / 2) * P.N * 128 * sizeof(float);
}

cudaError_t split_x_to_boxes(int in_dtype, const void* X, void* out, int64_t n, int32_t p, int32_t p_pad, int* err,
                             cudaStream_t s) {
  const int64_t nfb = p_pad / split::kBlk, blocks = (n + split::kBlk - 1) / split::kBlk * nfb;
  if (blocks > int64_t(0x7fffffff)) return cudaErrorInvalidValue;
  if (in_dtype == HMC_F64)
    split::rows_to_boxes_kernel<double><<<unsigned(blocks), 256, 0, s>>>(static_cast<const double*>(X),
                                                                         static_cast<float*>(out), n, p, nfb, err);
  else
    split::rows_to_boxes_kernel<float><<<unsigned(blocks), 256, 0, s>>>(static_cast<const float*>(X),
                                                                        static_cast<float*>(out), n, p, nfb, err);
  return cudaGetLastError();
}

cudaError_t split_boxes_to_rows(const void* boxes, void* out, int64_t n, int32_t p, int32_t p_pad, cudaStream_t s) {
  split::boxes_to_rows_kernel<<<4096, 256, 0, s>>>(static_cast<const float*>(boxes), static_cast<float*>(out), n, p,
                                                   p_pad / split::kBlk);
  return cudaGetLastError();
}

cudaError_t split_launch(const SplitPlan& P, const SplitLaunch& L, cudaStream_t s, cudaEvent_t between, bool capturing) {
  if (L.C < 1 || L.C > P.N) return cudaErrorInvalidValue;
  const int N = split_columns(L.C);
  const int64_t ta = (P.nrb + 1) / 2, tb = (P.nfb + 1) / 2;
  {
    const int64_t total = int64_t(L.C) * (P.p_pad / 8);
    const cudaError_t e = launch_chained(split::coef_boxes_kernel, unsigned(std::min<int64_t>(2048, (total + 255) / 256)),
                                         256, 0, s, L.beta, static_cast<unsigned char*>(L.bbox), L.C, N, P.p_pad);
    if (e != cudaSuccess) return e;
  }
  split::Args a{};
  a.xs = static_cast<const unsigned char*>(L.X);
  a.err = L.err;
  a.nrb = P.nrb;
  a.nfb = P.nfb;
  a.N = N;
  a.C = L.C;
  a.p_pad = P.p_pad;
  a.nstx = P.nstx;
  a.nstb = P.nstb;
  a.spin_limit = L.spin_limit;
  a.bs = static_cast<const unsigned char*>(L.bbox);
  a.out = L.zpart;
  a.out_stride = ta * N * 128;
  a.keep_rb = split::kKeepBytes / (P.nfb * split::kBoxBytes);
  a.ntiles = ta;
  a.groups = 1;
  a.ksteps = P.nfb;
  a.nslots = P.slotsA;
  cudaError_t e = launch_chained(split_gemm(false, N), P.gridA, split::kThreads, P.smem, s, a);
  if (e != cudaSuccess) return e;
  e = launch_chained(split::softmax_kernel, unsigned(P.nrb), split::kSoftThreads, split::softmax_smem(L.C, L.chains), s,
                     L.zpart, a.out_stride, L.y, static_cast<unsigned char*>(L.rbox), L.lrow, L.lrow_stride, L.n, L.C, N,
                     L.Km1, L.chains, L.zlogit, P.nfb, ta * P.nfb, P.gridA, L.err);
  if (e != cudaSuccess) return e;
  if (between) {
    e = capturing ? cudaEventRecordWithFlags(between, s, cudaEventRecordExternal) : cudaEventRecord(between, s);
    if (e != cudaSuccess) return e;
  }
  a.bs = static_cast<const unsigned char*>(L.rbox);
  a.out = L.gpart;
  a.out_stride = L.gpart_cstride;
  a.ntiles = tb;
  a.ksteps = P.nrb;
  a.nslots = P.slotsB;
  return launch_chained(split_gemm(true, N), P.gridB, split::kThreads, P.smem, s, a);
}

// The general kernel (one warp per row, one load per multiply) takes about 0.6 us per
// draw and 32 features of a row one after the other, and 1.5e6 multiplies per us over
// all rows; this path has a fixed cost of about 100 us (five launches and a
// synchronisation) and forms the boxes of X.  Measured, general -> this path: 10 rows
// p=785 K=10 100 draws 1398 -> 95 us, 10000 rows 4308 -> 267 us, 20000 rows p=2000
// K=20 200 draws 306 -> 3.7 ms; 20000 rows p=785 1 draw (107 us; here 145) and 1000 rows
// p=100 20 draws (85 us) stay.
bool split_predict_pays(int64_t n, int64_t p, int32_t km1, int64_t ndraws) {
  const double general = 0.6 * double(ndraws) * double((p + 31) / 32) + double(n) * double(p) * km1 * double(ndraws) / 1.5e6;
  return general >= 100.0 + double(n) * double(p) / 3e5;
}

// The rows and draws of one round, within `budget` bytes of scratch: up to 16384
// rows, then as many groups of draws as the logits leave room for.  No plan (groups 0)
// where the boxes of these rows alone fill the budget: with 256 MB, p above about 3900 at
// 16384 rows, 6400 at 10000; such calls stay with the general kernel.
SplitPredictPlan split_predict_plan(int64_t n, int64_t p, int32_t km1, int64_t ndraws, int nsm, int smem_max,
                                    size_t budget) {
  SplitPredictPlan P{};
  P.rows = std::min<int64_t>((n + 127) / 128 * 128, 16384);
  P.dpg = std::max(1, kSplitMaxN / km1);
  P.dpg = int(std::min<int64_t>(P.dpg, ndraws));
  const int C = P.dpg * km1;
  SplitPlan sp;
  if (!split_plan(P.rows, p, C, nsm, smem_max, &sp)) return P;
  const int64_t tiles = P.rows / 128, all = (ndraws + P.dpg - 1) / P.dpg;
  P.xbytes = split_x_bytes(sp);
  const size_t gbytes = split_box_bytes(sp, sp.nfb), unit = size_t(sp.N) * 128 * sizeof(float);
  const size_t fixed = P.xbytes + size_t(P.rows) * 32 * sizeof(double) + 256;
  P.rows_pad = P.rows;
  for (int64_t g = all; g >= 1; g = g > 1 ? (g + 1) / 2 : 0) {
    // A launch of u units on G CTAs has at most ksteps G / W + 2 = G / u + 2 partials
    // per unit, so this holds the logits of every round, full or not.
    const size_t zbytes = size_t(2 * g * tiles + nsm) * unit;
    const size_t kbytes = size_t(g) * P.dpg * P.rows * sizeof(float);   // probabilities of class K
    const size_t total = fixed + size_t(g) * gbytes + zbytes + kbytes;
    if (total <= budget) {
      P.groups = g;
      P.grid = nsm;
      P.bbytes = size_t(g) * gbytes;
      P.zbytes = zbytes;
      P.kbytes = kbytes;
      P.total = total;
      P.sp = sp;
      break;
    }
  }
  return P;
}

cudaError_t split_predict(const SplitPredictPlan& P, int in_dtype, const void* X, int64_t n, int32_t p, const float* draws,
                          int64_t ndraws, int32_t ku, int32_t km1, int32_t zlogit, int32_t K, double* prob, int32_t* cls,
                          void* scratch, int* flag, int* err, long long spin_limit, cudaStream_t s) {
  unsigned char* xb = static_cast<unsigned char*>(scratch);
  unsigned char* bb = xb + P.xbytes;
  float* z = reinterpret_cast<float*>(bb + P.bbytes);
  float* pk = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(z) + P.zbytes);
  double* acc = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(pk) + P.kbytes);
  const int64_t nfb = P.sp.nfb;
  const size_t xrow = size_t(p) * (in_dtype == HMC_F64 ? 8 : 4);
  for (int64_t r0 = 0; r0 < n; r0 += P.rows) {
    const int64_t rows = std::min(P.rows, n - r0);
    cudaError_t e = split_x_to_boxes(in_dtype, static_cast<const char*>(X) + size_t(r0) * xrow, xb, rows, p, P.sp.p_pad,
                                     flag, s);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (rows + 127) / 128;
    for (int64_t d0 = 0; d0 < ndraws; d0 += P.groups * P.dpg) {
      const int64_t nd = std::min(P.groups * P.dpg, ndraws - d0);
      const int64_t g = (nd + P.dpg - 1) / P.dpg;
      const int64_t work = nd * km1 * (P.sp.p_pad / 8);
      split::draw_boxes_kernel<<<unsigned(std::min<int64_t>(4096, (work + 255) / 256)), 256, 0, s>>>(
          draws + size_t(d0) * ku * p, bb, nd, ku, km1, p, P.sp.p_pad, P.dpg, P.sp.N, flag);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      split::Args a{};
      a.xs = xb;
      a.bs = bb;
      a.out = z;
      a.err = err;
      a.nrb = (rows + split::kBlk - 1) / split::kBlk;
      a.nfb = nfb;
      a.ntiles = tiles;
      a.keep_rb = split::kKeepBytes / (nfb * split::kBoxBytes);
      a.groups = int32_t(g);
      a.ksteps = int32_t(nfb);
      a.N = P.sp.N;
      a.C = P.dpg * km1;
      a.p_pad = P.sp.p_pad;
      a.nstx = P.sp.nstx;
      a.nstb = P.sp.nstb;
      a.spin_limit = spin_limit;
      a.out_stride = g * tiles * P.sp.N * 128;
      const int64_t W = g * tiles * nfb;
      if (W > int64_t(0x7fffffff)) return cudaErrorInvalidValue;
      // At most four CTAs to a unit: more partials cost the next kernel more.
      const int64_t grid = std::min<int64_t>({P.grid, W, 4 * g * tiles});
      a.nslots = int32_t(split_slots(g * tiles, nfb, grid));
      if (size_t(a.nslots) * a.out_stride * sizeof(float) > P.zbytes) return cudaErrorInvalidValue;
      split_gemm(false, P.sp.N)<<<unsigned(grid), split::kThreads, P.sp.smem, s>>>(a);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      auto launch = [&](auto kb) {
        split::predict_prob_kernel<decltype(kb)::value><<<unsigned(g * tiles * P.dpg), 128, 0, s>>>(
            z, a.out_stride, tiles, P.sp.N, nfb, W, grid, rows, nd, P.dpg, km1, zlogit, pk, P.rows_pad, flag);
      };
      if (km1 <= 4) launch(std::integral_constant<int, 4>{});
      else if (km1 <= 10) launch(std::integral_constant<int, 10>{});
      else if (km1 <= 20) launch(std::integral_constant<int, 20>{});
      else launch(std::integral_constant<int, 32>{});
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      split::predict_sum_kernel<<<unsigned((rows + 31) / 32), dim3(32, K), 0, s>>>(
          z, tiles, P.sp.N, rows, nd, P.dpg, km1, K, pk, P.rows_pad, acc, d0 == 0 ? 1 : 0,
          d0 + nd == ndraws ? double(ndraws) : 0.0, prob ? prob + size_t(r0) * K : nullptr, cls ? cls + r0 : nullptr);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

}  // namespace hmc
