// Fused log-posterior + gradient pass on the 5th-generation tensor cores
// (tcgen05) for X stored in BF16 or per-column-scaled FP8 (widened to BF16 in
// shared memory), many chains at once (Eqs. softmax, loglike,
// logkernel and gradient of Sec. 2.1, evaluated for C = chains*(K-1)
// coefficient columns).
//
// Decomposition: a cluster of S CTAs walks row tiles of 128 rows; CTA `rank`
// owns the column slice [rank*PC, (rank+1)*PC) (PC a multiple of 128) of X and
// of the coefficients, and accumulates the gradient rows of that slice in
// TMEM across all of the cluster's tiles.  Per tile:
//   sweep 1  bulk-async copies bring 128 x 64 boxes of X together with the
//            matching 64-column box of the coefficients as two BF16 terms
//            (B = B_hi + B_lo); MMAs D_z[128 x N] += X_box . B_hi^T and
//            += X_box . B_lo^T (both operands K-major), so the logits carry
//            the coefficients to ~16 bits.
//            X and the coefficient operand are stored in device memory as
//            the shared-memory image of these boxes (128-byte swizzle already
//            applied, each box 16 KB contiguous), so every copy is a long
//            contiguous read.
//   exchange (distributed shared memory only) the drain warps read D_z, one
//            row per thread, and push each row with st.async into the shared
//            memory of the CTA that owns it (rows are split 128/S per CTA);
//            the owner sums the S partials in rank order, forms the softmax
//            with the zero logit of class K, the residual R = Y - P (BF16) and
//            the row log-likelihood, and pushes its R rows with st.async
//            straight into every peer's MMA operand buffer (swizzled layout).
//            Completion is counted in mbarrier transaction bytes.
//   sweep 2  X is re-read in 128-column blocks (an L2 hit: the tile was
//            streamed one sweep earlier); MMA D_g[mb] (128 columns x N) +=
//            X_blk^T . R with X_blk read MN-major from the same swizzled boxes
//            and R MN-major from the operand buffer.  The commit of these MMAs
//            is multicast to every CTA of the cluster, telling the owners
//            that the R buffer may take the rows of a later tile.
// Sweeps are interleaved S1(0), S1(1), S2(0), S1(2), S2(1), ... so the
// exchange of one tile overlaps the next tile's first sweep: in one line of ring
// slots, in that order, or in two lines, each with a producer and an MMA issuer, where
// sweep 1 keeps the same distance from sweep 2 (ring_lines).
// What bounds it: the copies from L2, which hands X out twice and the coefficients once
// a tile.  32 problems of uneven size in BF16, C = 4 .. 19 (1.25 GB of X, 2.9 GB copied):
// 1073 us with a cluster per problem at least, 529 us with the clusters' work in items of
// equal cost, 465 us with the softmax and the issue of MMAs made cheaper, 370 us with two
// lines (7.8 TB/s).  n=4e5 p=1500 C=9: 515 -> 263 us, n=1.5e5 p=4000 C=19: 508 -> 347 us
// in BF16, 836 -> 565 us in FP8, whose slots wait for the converters.
// Warp roles: warp 0 TMA producer (lane 0 alone: no other role shares its
// warp, so nothing suspends the copy issue), warp 1 TMEM owner + MMA issuer,
// warps 2-5 drain group (TMEM lanes 0-127; the gradient slice at the end),
// warps 6-13 softmax group, warps 14-21 FP8 converters (FP8 X only), the last
// two warps producer and MMA issuer of line 1.  All waits are bounded.
#include <algorithm>
#include <vector>
#include <cstring>

#include "internal.h"
#include "tc_common.cuh"

namespace hmc {
namespace tc {

constexpr int kThreadsBf16 = 512;   // warps 0-13, and the last two: line 1
constexpr int kThreadsFp8 = 768;    // + warps 14-21 (FP8 converters), and the last two: line 1
constexpr int kSoftThreads = 256;   // warps 6-13
constexpr int kConvWarps = 8;       // warps 14-21: FP8 -> BF16 converters (FP8 X only)
constexpr int kConvThreads = 32 * kConvWarps;
constexpr int kFp8BoxBytes = 128 * 64;   // one FP8 box: 128 rows x 64 bytes, row-major
constexpr int kMaxDepth = kTcMaxDepth;   // largest number of logit accumulators / exchange slots / R buffers
constexpr int kRows = 128;
constexpr int kBox = 64;          // BF16 elements per 128-byte box row
constexpr int kBoxBytes = kRows * 128;
constexpr int kMaxAhead = 7;      // sweeps 1 ahead of sweep 2, at most, with two lines

struct TcArgs {
  const void* xs;           // X boxes, [row tile][p_pad / 64][box]: BF16 in its swizzled shared-memory
                            // image (16 KB), or FP8 E4M3 row-major (8 KB) when fp8
  const float* xscale;      // FP8: per-column scales s_j (X = X_q diag(s)); nullptr for BF16
  const __nv_bfloat16* bs;  // coefficient operand boxes: [p_pad / 64][N rows x 128 B]
  int64_t n;
  int32_t p_pad, PC, S, N, NP, C, Km1, chains, MB, NST, nclusters;
  int64_t ntiles;
  uint32_t tmem_cols, stage_bytes;
  float* gpart;             // [cluster][C][p_pad] partial gradient (this launch's columns)
  int64_t gpart_cstride;
  double* lpart;            // [cluster*S + rank][lpart_cstride] partial log-likelihood per chain
  int32_t lpart_cstride;
  const int32_t* y;
  int* err;
  long long spin_limit;
  int32_t inject_timeout;
  int32_t fp8;
  int32_t zlogit;           // 1: class K is the implied zero logit; 0: all Km1 classes free
  // Pipeline depths (host-chosen from the TMEM and shared-memory budgets):
  int32_t nz;      // logit accumulators in TMEM (sweep 1 of the next tiles runs while one drains)
  int32_t slots;   // partial-logit receive slots (reuse gated by a cluster 'consumed' barrier)
  int32_t rbufs;   // R operand buffers (reuse gated by a cluster 'free' barrier)
  int32_t la;      // tiles of lookahead between the two sweeps of a tile
};

// The shared-memory ring of `nst` x `stage_bytes` as one line of slots for both sweeps,
// or as two lines: sweep 1 (X box and coefficient box) with n0 slots of b0 bytes, sweep 2
// (two X boxes) with n1 slots of 32 KB behind them.  Two lines want two slots of sweep 2
// and one more of sweep 1 at least: with 2 + 2 slots (C = 17 .. 32 in 128 KB) 32 uneven
// problems took 445 us against 405 with these in one line; 6 + 2 slots in 192 KB were
// slower than 4 + 3 (28000 and 24000 clocks a tile of 26 boxes).
struct Lines {
  int two, n0, n1;
  uint32_t b0, off1;
};
__host__ __device__ inline Lines ring_lines(int nst, uint32_t stage_bytes, int N) {
  Lines L{0, nst, 0, stage_bytes, 0};
  const uint32_t ring = uint32_t(nst) * stage_bytes, b1 = 2 * kBoxBytes;
  const uint32_t b0 = (uint32_t(kBoxBytes) + uint32_t(2 * N) * 128u + 1023u) / 1024u * 1024u;
  int n1 = 2;
  while (ring >= uint32_t(n1 + 1) * b1 + uint32_t(n1 + 2) * b0) ++n1;
  if (ring < uint32_t(n1) * b1 + uint32_t(n1 + 1) * b0) return L;
  L.two = 1;
  L.n1 = n1;
  L.n0 = int((ring - uint32_t(n1) * b1) / b0);
  L.b0 = b0;
  L.off1 = uint32_t(L.n0) * b0;
  return L;
}

struct Smem {
  size_t ring, stage, rbuf, zx, rloc, lacc, ylab, bars, total;
};

__host__ __device__ inline size_t al(size_t v, size_t a) { return (v + a - 1) / a * a; }

// zx: [slots][S][RS][N] fp32 partial logits received for the owned rows, the 16-byte
// chunks of a row permuted by zx_swizzle; rloc: [RS][NP] bf16 residual rows of the owned
// rows before they are pushed, the chunks of each 128 bytes of row r permuted by ^ r % 8.
__host__ __device__ inline Smem smem_layout(int NST, uint32_t stage_bytes, int NP, int N, int S, int chains, bool fp8,
                                            int slots, int rbufs) {
  Smem L;
  const int RS = kRows / S;
  size_t off = 0;
  L.ring = off;  off = al(off + size_t(NST) * stage_bytes, 1024);
  // FP8 boxes land in the upper half of their slot's X area and are widened in place.
  L.stage = off;
  L.rbuf = off;  off = al(off + size_t(rbufs) * (NP / kBox) * kBoxBytes, 1024);
  L.zx = off;    off = al(off + size_t(slots) * kRows * N * 4, 16);
  L.rloc = off;  off = al(off + size_t(RS) * NP * 2, 16);
  L.lacc = off;  off = al(off + size_t(RS) * chains * 8, 16);
  L.ylab = off;  off = al(off + size_t(RS) * 4, 16);
  const Lines ln = ring_lines(NST, stage_bytes, N);
  L.bars = off;  off = al(off + size_t(3 * (ln.n0 + ln.n1) + 6 * kMaxDepth + kMaxAhead + 1 + 7) * 8 + 16, 16);
  L.total = off + 1024;  // slack for aligning the dynamic base to 1024
  return L;
}

__device__ __forceinline__ bool wait_bounded(uint64_t* bar, uint32_t parity, long long limit, volatile int* abort,
                                             bool cluster_scope) {
  const uint32_t a = smem_u32(bar);
  for (long long i = 0; i < limit; ++i) {
    if (cluster_scope ? mbar_test_cluster(a, parity) : mbar_test_cta(a, parity)) return true;
    if ((i & 63) == 63 && *abort) return false;
  }
  return false;
}

// Chunk c of row r of zx sits at chunk c ^ zx_swizzle(r, N): eight consecutive rows
// then hold a class in eight different bank groups (N is a multiple of 16, so a row
// starts at bank 0, or at bank 0 or 16 in turn).
__device__ __forceinline__ int zx_swizzle(int r, int N) { return (N & 16) ? (r >> 1) & 3 : r & 7; }

__device__ __forceinline__ void named_bar_soft() { asm volatile("bar.sync 2, 256;" ::: "memory"); }
// Barrier of one of the FP8 converter groups (named barrier 3 + group, n threads), and the
// same barrier ANDing a flag across the group (so every converter leaves its loop together).
__device__ __forceinline__ void conv_bar(int g, int n) { asm volatile("bar.sync %0, %1;" ::"r"(3 + g), "r"(n) : "memory"); }
__device__ __forceinline__ bool conv_bar_and(int g, int n, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "bar.red.and.pred po, %2, %3, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "r"(3 + g), "r"(n)
      : "memory");
  return r != 0;
}
// Named barrier of the softmax group that also ANDs a flag across its threads.
__device__ __forceinline__ bool named_bar_soft_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "bar.red.and.pred po, 2, 256, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u)
      : "memory");
  return r != 0;
}

// What one cluster does of a problem: tiles tile0 + u * tstride, u < tiles; its
// partials go to slot `slot`.
struct TcShare {
  int64_t tile0, tstride, tiles;
  int32_t slot;
};

// One cluster's share of the fused pass for problem A.  `base` is the TMEM the
// kernel allocated; nullptr: the body allocates what it needs.  `stop`: raised in
// every CTA of the cluster if a wait ran out (nullptr: a word of the body's own).
template <bool kFP8>
__device__ __forceinline__ void tc_body(const TcArgs& A, const TcShare& W, const uint32_t* base, int* stop) {
  constexpr int kThreads = kFP8 ? kThreadsFp8 : kThreadsBf16;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int S = A.S, N = A.N, NP = A.NP;
  const Lines ln = ring_lines(A.NST, A.stage_bytes, N);
  const bool two = ln.two != 0;
  const int nslots = ln.n0 + ln.n1;
  const uint32_t rank = (S > 1) ? cluster_rank() : 0u;
  const int RS = kRows / S;                        // rows this CTA owns in the exchange
  const int chains = A.chains, C = A.C, Km1 = A.Km1;
  const bool zl = A.zlogit != 0;
  const int C8 = (C + 7) / 8;                      // 16-byte chunks of one R row
  constexpr bool fp8 = kFP8;
  const int NZ = A.nz, SLOTS = A.slots, RBUFS = A.rbufs, LA = two && A.la > kMaxAhead ? kMaxAhead : A.la;
  const Smem Lo = smem_layout(A.NST, A.stage_bytes, NP, N, S, chains, fp8, SLOTS, RBUFS);
  unsigned char* ring = smem + Lo.ring;
  unsigned char* rbuf = smem + Lo.rbuf;
  float* zx = reinterpret_cast<float*>(smem + Lo.zx);
  __nv_bfloat16* rloc = reinterpret_cast<__nv_bfloat16*>(smem + Lo.rloc);
  double* lacc = reinterpret_cast<double*>(smem + Lo.lacc);
  int* ylab = reinterpret_cast<int*>(smem + Lo.ylab);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lo.bars);
  uint64_t* full = bars;
  uint64_t* empty = bars + nslots;
  uint64_t* conv = bars + 2 * nslots;      // FP8: ring slot converted to BF16 (an arrival per converter warp)
  uint64_t* zdone = bars + 3 * nslots;        // [nz] sweep 1 of a tile finished in accumulator z
  uint64_t* zfree = zdone + kMaxDepth;      // [nz] accumulator z drained
  uint64_t* zrdy = zfree + kMaxDepth;       // [slots] partial logits of the owned rows received
  uint64_t* zxfree = zrdy + kMaxDepth;      // [slots] every owner has consumed the slot's partials
  uint64_t* rfull = zxfree + kMaxDepth;     // [rbufs] every owner's R rows received (R buffer b)
  uint64_t* rfreec = rfull + kMaxDepth;     // [rbufs] every CTA's gradient sweep finished reading R buffer b
  uint64_t* ahead_bar = rfreec + kMaxDepth; // [LA + 1] two lines: sweep 2 of a tile issued and complete
  uint64_t* gdone = ahead_bar + kMaxAhead + 1;
  uint64_t* drain = gdone + 1;              // [2] a line's MMAs are complete
  uint64_t* never = gdone + 3;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gdone + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gdone + 5);
  if (!stop) stop = reinterpret_cast<int*>(gdone + 6);
  const size_t rbuf_bytes = size_t(NP / kBox) * kBoxBytes;

  if (tid == 0) {
    for (int s = 0; s < nslots; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&conv[s], two ? kConvWarps / 2 : kConvWarps);
    }
    for (int b = 0; b <= kMaxAhead; ++b) mbar_init(&ahead_bar[b], 1);
    for (int b = 0; b < kMaxDepth; ++b) {
      mbar_init(&zdone[b], 1);
      mbar_init(&zfree[b], 4);
      mbar_init(&zrdy[b], 1);
      mbar_init(&zxfree[b], S);
      mbar_init(&rfull[b], 1);
      mbar_init(&rfreec[b], S);
    }
    mbar_init(gdone, 1);
    mbar_init(&drain[0], 1);
    mbar_init(&drain[1], 1);
    mbar_init(never, 1);
    *abort_flag = 0;
    *stop = 0;
    fence_mbar_init_cluster();
  }
  // R operand buffer and the local R rows start (and stay, past column C) zero.
  for (size_t i = tid; i < RBUFS * rbuf_bytes / 16; i += kThreads)
    reinterpret_cast<uint4*>(rbuf)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < RS * NP / 8; i += kThreads) reinterpret_cast<uint4*>(rloc)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < RS * chains; i += kThreads) lacc[i] = 0.0;
  fence_proxy_async_smem();
  if (warp == 1 && !base) tmem_alloc(tmem_slot, A.tmem_cols);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = base ? *base : *tmem_slot;
  if (A.inject_timeout && tid == 0) {
    if (!wait_bounded(never, 0u, A.spin_limit, abort_flag, false)) {
      *abort_flag = 1;
      atomicOr(A.err, ERR_TIMEOUT_STAGE);
    }
  }
  if (S > 1)
    cluster_sync_all();
  else
    __syncthreads();

  const int64_t T = *abort_flag ? 0 : W.tiles;
  const int64_t nphase = 2 * T;
  const int NKB = A.PC / kBox;
  const int64_t nkb_all = A.p_pad / kBox;
  // Phase k of the sweep order: S1(0..first-1), then pairs S1(v), S2(v-la),
  // then the remaining S2 phases.  Returns the tile; *s2 marks a gradient sweep.
  const int64_t first = T < LA ? T : LA;
  auto phase = [&](int64_t k, bool* s2) -> int64_t {
    if (k < first) { *s2 = false; return k; }
    const int64_t k1 = k - first;
    if (k1 < 2 * (T - first)) {
      *s2 = (k1 & 1) != 0;
      return *s2 ? (k1 >> 1) : first + (k1 >> 1);
    }
    *s2 = true;
    return T - first + (k1 - 2 * (T - first));
  };
  auto fail = [&](int bit) {
    *abort_flag = 1;
    atomicOr(A.err, bit);
  };

  // The two sweeps share one line of ring slots, in the order of the phases; with enough
  // slots each sweep has a line, a producer and an issuer of its own, so that one's
  // waits pass while the other's MMAs run.
  constexpr int kLine1 = kThreads / 32 - 2;
  const int line = warp >= kLine1 ? 1 : 0;
  const int nring = line ? ln.n1 : ln.n0;
  const uint32_t slot_bytes = line ? 2u * kBoxBytes : ln.b0;
  unsigned char* const lring = ring + (line ? ln.off1 : 0u);
  auto mine = [&](bool s2) { return two ? s2 == (line != 0) : line == 0; };
  if (warp == 0 || warp == kLine1) {
    // ---------------------------------------------------------------- TMA producers
    if (lane == 0) {
      int64_t j = 0, issued = 0;
      Ring r;
      full += line * ln.n0;
      empty += line * ln.n0;
      for (int64_t k = 0; k < nphase && !*abort_flag; ++k) {
        bool s2;
        const int64_t u = phase(k, &s2);
        if (!mine(s2)) continue;
        const int nb = s2 ? A.MB : NKB;
        for (int b = 0; b < nb; ++b, ++j, r.next(nring)) {
          const int st = r.slot;
          if (!wait_bounded(&empty[st], r.par ^ 1u, A.spin_limit, abort_flag, false)) {
            fail(ERR_TIMEOUT_STAGE);
            break;
          }
          unsigned char* sp = lring + size_t(st) * slot_bytes;
          const int64_t t = W.tile0 + u * W.tstride;  // row tile
          const uint32_t xbox = fp8 ? uint32_t(kFp8BoxBytes) : uint32_t(kBoxBytes);
          const unsigned char* xt = reinterpret_cast<const unsigned char*>(A.xs) + size_t(t) * nkb_all * xbox;
          // BF16 X lands in the slot itself; FP8 X lands in the upper half of the
          // slot's X area and the converter warps widen it in place.
          unsigned char* xdst = fp8 ? sp + size_t(s2 ? 2 : 1) * (kBoxBytes - kFp8BoxBytes) : sp;
          if (!s2) {
            const int kb = int(rank) * NKB + b;
            mbar_arrive_expect_tx(&full[st], xbox + uint32_t(2 * N * 128));
            bulk_g2s(xdst, xt + size_t(kb) * xbox, xbox, &full[st]);
            bulk_g2s(sp + kBoxBytes, reinterpret_cast<const unsigned char*>(A.bs) + size_t(kb) * 2 * N * 128,
                     uint32_t(2 * N * 128), &full[st]);
          } else {
            const int kb = int(rank) * NKB + 2 * b;
            mbar_arrive_expect_tx(&full[st], 2 * xbox);
            bulk_g2s(xdst, xt + size_t(kb) * xbox, 2 * xbox, &full[st]);
          }
          issued = j + 1;
        }
      }
      // Every copy issued must land before shared memory is released.
      for (int64_t jj = (issued > nring ? issued - nring : 0); jj < issued; ++jj)
        wait_drain(&full[jj % nring], uint32_t((jj / nring) & 1), A.spin_limit);
    }
  } else if (warp == 1 || warp == kLine1 + 1) {
    // ---------------------------------------------------------------- MMA issuers
    // The whole warp runs the loop (waits included), one elected lane issues.
    const uint32_t id_s1 = uniform(idesc_bf16(kRows, N, false, false));
    const uint32_t id_s2 = uniform(idesc_bf16(kRows, N, true, true));
    const uint32_t tm = uniform(tmem), nu = uniform(uint32_t(N));
    const uint32_t rg = uniform(desc_addr(lring)), rb = uniform(desc_addr(rbuf));
    const uint32_t sbytes = uniform(slot_bytes >> 4), rbsize = uniform(uint32_t(rbuf_bytes >> 4));
    const uint64_t desc1 = smem_desc(0u, 16u, 1024u, 2u), desc2 = smem_desc(0u, uint32_t(kBoxBytes), 1024u, 2u);
    const uint32_t rbytes = uint32_t(kRows) * C8 * 16;
    const int MB = A.MB;
    const long long limit = A.spin_limit;
    uint64_t* ready = (fp8 ? conv : full) + line * ln.n0;
    empty += line * ln.n0;
    Ring r, zr, rr, ar;                     // ring slot, logit accumulator, R buffer, tiles ahead
    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t parity, bool cluster_scope, int bit) {
      ok = __all_sync(0xffffffffu, wait_bounded(bar, parity, limit, abort_flag, cluster_scope));
      if (!ok && lane == 0) fail(bit);
      return ok;
    };
    // The next slot is looked at before the MMAs of this one go out: the tensor pipe
    // takes one MMA at a time (40 clocks each at N = 16, reading A), so a wait that
    // starts after the last of them leaves it idle for all of its 150 clocks or more.
    bool ahead = false;
    auto wait_slot = [&]() {
      if (__all_sync(0xffffffffu, ahead)) return true;
      return wait(&ready[r.slot], r.par, false, ERR_TIMEOUT_STAGE);
    };
    auto look = [&]() {
      Ring n = r;
      n.next(nring);
      ahead = mbar_look_cta(smem_u32(&ready[n.slot]), n.par) && limit > 0;
    };
    for (int64_t k = 0; k < nphase && ok; ++k) {
      bool s2;
      const int64_t u = phase(k, &s2);
      if (!mine(s2)) continue;
      if (!s2) {
        // Two lines: sweep 1 stays as far ahead of sweep 2 as with one, or the rows of X
        // would have left L2 before their second use.  (Sweep 2 cannot pass sweep 1, so
        // a barrier of the ring of LA + 1 is one use ahead of this wait at most.)
        if (two && u > LA) {
          if (!wait(&ahead_bar[ar.slot], ar.par, false, ERR_TIMEOUT_MMA)) break;
          ar.next(LA + 1);
        }
        // Accumulator z = u % nz was last used by tile u - nz: it must be drained.
        if (u >= NZ && !wait(&zfree[zr.slot], zr.par ^ 1u, false, ERR_TIMEOUT_MMA)) break;
        const uint32_t dz = uniform(tm + uint32_t(zr.slot) * nu);
        fence_after_sync();
        for (int kb = 0; kb < NKB; ++kb, r.next(nring)) {
          if (!wait_slot()) break;
          fence_after_sync();
          look();
          const uint64_t xd = desc1 | uniform(rg + uint32_t(r.slot) * sbytes);
          if (elect_one()) {
            const uint64_t bd = xd + uint64_t(kBoxBytes >> 4), bl = bd + nu * 8u;   // hi rows; lo rows N * 128 bytes further
#pragma unroll
            for (int s = 0; s < 4; ++s) {
              mma_bf16(dz, xd + 2u * s, bd + 2u * s, id_s1, (kb > 0 || s > 0) ? 1u : 0u);
              mma_bf16(dz, xd + 2u * s, bl + 2u * s, id_s1, 1u);
            }
            mma_commit(&empty[r.slot]);
            if (kb == NKB - 1) mma_commit(&zdone[zr.slot]);
          }
          __syncwarp();
        }
        zr.next(NZ);
      } else {
        if (elect_one()) mbar_arrive_expect_tx(&rfull[rr.slot], rbytes);
        __syncwarp();
        if (!wait(&rfull[rr.slot], rr.par, true, ERR_TIMEOUT_EXCHANGE)) break;
        fence_after_sync();
        const uint64_t rd = desc2 | uniform(rb + uint32_t(rr.slot) * rbsize);
        for (int mb = 0; mb < MB; ++mb, r.next(nring)) {
          if (!wait_slot()) break;
          fence_after_sync();
          look();
          const uint64_t xd = desc2 | uniform(rg + uint32_t(r.slot) * sbytes);
          const uint32_t dcol = uniform(tm + uint32_t(NZ + mb) * nu);
          if (elect_one()) {
#pragma unroll
            for (int s = 0; s < 8; ++s) mma_bf16(dcol, xd + 128u * s, rd + 128u * s, id_s2, (u > 0 || s > 0) ? 1u : 0u);
            mma_commit(&empty[r.slot]);
            if (two && mb == MB - 1) mma_commit(&ahead_bar[ar.slot]);
            // This R buffer is free once these MMAs complete: the commit arrives on
            // that buffer's barrier in every CTA of the cluster, so each owner may
            // push the R rows of tile u + rbufs.  Only tiles whose buffer is used
            // again signal, so every remote arrival has a waiter in its CTA (and
            // lands before that CTA can leave the kernel).
            if (mb == MB - 1 && u + RBUFS < T) {
              if (S > 1)
                mma_commit_multicast(&rfreec[rr.slot], uint16_t((1u << S) - 1u));
              else
                mma_commit(&rfreec[rr.slot]);
            }
          }
          __syncwarp();
        }
        rr.next(RBUFS);
        ar.next(LA + 1);
      }
    }
    if (elect_one()) {
      if (line == (two ? 1 : 0)) mma_commit(gdone);
      mma_commit(&drain[line]);
    }
    __syncwarp();
    wait_drain(&drain[line], 0u, limit);
  } else if (kFP8 && warp >= 14) {   // the last two warps are taken above
    // --------------------------------------- FP8 converters (warps 14-21)
    // Each FP8 box (128 rows x 64 bytes, landed in the upper half of its
    // slot's X area) is widened to BF16 (exact: every E4M3 value is a BF16
    // value) and written over the slot in the 128-byte-swizzled layout the
    // MMAs read; sweep-2 slots hold two boxes.  Every converter thread reads
    // all its input chunks before a converter-group barrier and only then
    // writes, so the in-place widening never overwrites unread input.  With two
    // lines the warps are two groups, one for each.
    {
      const int nconv = two ? kConvThreads / 2 : kConvThreads;
      const int cg = (tid - 448) / nconv, ct = (tid - 448) % nconv;   // group, thread of the group
      const int nring = cg ? ln.n1 : ln.n0;
      const uint32_t slot_bytes = cg ? 2u * kBoxBytes : ln.b0;
      unsigned char* const lring = ring + (cg ? ln.off1 : 0u);
      full += cg * ln.n0;
      conv += cg * ln.n0;
      Ring rr;
      bool ok = true;
      for (int64_t k = 0; k < nphase && ok; ++k) {
        bool s2;
        (void)phase(k, &s2);
        if (two && s2 != (cg != 0)) continue;
        const int nb = s2 ? A.MB : NKB;
        const int nbox = s2 ? 2 : 1;
        const int per = nbox * (kFp8BoxBytes / 16) / nconv;   // chunks per thread
        for (int b = 0; b < nb; ++b, rr.next(nring)) {
          const int st = rr.slot;
          const bool got = wait_bounded(&full[st], rr.par, A.spin_limit, abort_flag, false);
          // Every converter agrees before the group barriers below.
          if (!conv_bar_and(cg, nconv, got && !*abort_flag)) {
            if (!got) fail(ERR_TIMEOUT_STAGE);
            ok = false;
            break;
          }
          unsigned char* dst = lring + size_t(st) * slot_bytes;
          const unsigned char* src = dst + size_t(nbox) * (kBoxBytes - kFp8BoxBytes);
          // Input chunk ci (16 bytes) of box bx: row ci / 4, elements 16 (ci % 4) ...
          constexpr int kPer = (2 * kFp8BoxBytes / 16) / (kConvThreads / 2);
          uint4 w[kPer];
#pragma unroll
          for (int i = 0; i < kPer; ++i)
            if (i < per) w[i] = *reinterpret_cast<const uint4*>(src + size_t(ct + nconv * i) * 16);
          conv_bar(cg, nconv);
#pragma unroll
          for (int i = 0; i < kPer; ++i) {
            if (i >= per) break;
            const int g = ct + nconv * i;                      // chunk over both boxes
            const int bx = g / (kFp8BoxBytes / 16), ci = g % (kFp8BoxBytes / 16);
            const int r = ci >> 2, qq = ci & 3;
            uint32_t o[8];
            fp8x4_to_bf16x4(w[i].x, o[0], o[1]);
            fp8x4_to_bf16x4(w[i].y, o[2], o[3]);
            fp8x4_to_bf16x4(w[i].z, o[4], o[5]);
            fp8x4_to_bf16x4(w[i].w, o[6], o[7]);
            unsigned char* rowp = dst + size_t(bx) * kBoxBytes + size_t(r) * 128;
            *reinterpret_cast<uint4*>(rowp + ((((2 * qq) ^ (r & 7))) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<uint4*>(rowp + ((((2 * qq + 1) ^ (r & 7))) << 4)) = make_uint4(o[4], o[5], o[6], o[7]);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive_local(&conv[st]);
        }
      }
    }
  } else if (warp < 6) {
    // ------------------------------------------------ drain group (warps 2-5)
    const int q = warp & 3;                 // TMEM lane quarter of this warp
    const int row = 32 * q + lane;          // tile row (sweep-1 accumulator lane)
    const uint32_t tq = tmem + (uint32_t(32 * q) << 16);
    const uint32_t owner = uint32_t(row / RS), rl = uint32_t(row % RS);
    const int zsw = zx_swizzle(int(rl), N);
    for (int64_t u = 0; u < T && !*abort_flag; ++u) {
      const int slot = int(u % SLOTS);
      const int z = int(u % NZ);
      // Lane 0 waits for each barrier and the warp follows it (one waiter per
      // warp keeps the barrier probes off the shared-memory pipe).
      bool ok = (lane == 0) ? wait_bounded(&zdone[z], uint32_t((u / NZ) & 1), A.spin_limit, abort_flag, false) : true;
      if (!__shfl_sync(0xffffffffu, ok, 0)) {
        if (lane == 0) fail(ERR_TIMEOUT_MMA);
        break;
      }
      fence_after_sync();
      // The owners' slot was last filled with tile u - slots: they must have consumed it.
      ok = (lane == 0 && u >= SLOTS)
               ? wait_bounded(&zxfree[slot], uint32_t(((u / SLOTS) - 1) & 1), A.spin_limit, abort_flag, true)
               : true;
      if (!__shfl_sync(0xffffffffu, ok, 0)) {
        if (lane == 0) fail(ERR_TIMEOUT_SLOT);
        break;
      }
      // This row's partial logits go to the owner's slot [slot][rank][rl].
      const uint32_t laddr = smem_u32(zx + ((size_t(slot) * S + rank) * RS + rl) * N);
      const uint32_t raddr = (S > 1) ? map_peer(laddr, owner) : laddr;
      const uint32_t rbar = (S > 1) ? map_peer(smem_u32(&zrdy[slot]), owner) : smem_u32(&zrdy[slot]);
      for (int c0 = 0; c0 < N; c0 += 16) {
        float v[16];
        tmem_ld16(tq + uint32_t(z * N + c0), v);
#pragma unroll
        for (int e = 0; e < 16; e += 4)
          st_async_v4f(raddr + uint32_t(((c0 + e) >> 2) ^ zsw) * 16u, v[e], v[e + 1], v[e + 2], v[e + 3], rbar);
      }
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_local(&zfree[z]);
    }
    // Drain the gradient accumulators of this CTA's column slice.
    bool gok = false;
    if (T > 0 && !*abort_flag) {
      gok = wait_bounded(gdone, 0u, A.spin_limit, abort_flag, false);
      if (!gok) fail(ERR_TIMEOUT_MMA);
    }
    float* gp = A.gpart + size_t(W.slot) * A.gpart_cstride;
    if (gok && !*abort_flag) {
      fence_after_sync();
      for (int mb = 0; mb < A.MB; ++mb) {
        const int col = int(rank) * A.PC + mb * 128 + row;
        const float sc = A.xscale ? A.xscale[col] : 1.0f;   // g = diag(s) X_q^T R
        for (int c0 = 0; c0 < N; c0 += 16) {
          float v[16];
          tmem_ld16(tq + uint32_t((NZ + mb) * N + c0), v);
#pragma unroll
          for (int e = 0; e < 16; ++e)
            if (c0 + e < C) gp[size_t(c0 + e) * A.p_pad + col] = v[e] * sc;
        }
      }
    } else {
      for (int mb = 0; mb < A.MB; ++mb) {
        const int col = int(rank) * A.PC + mb * 128 + row;
        for (int c = 0; c < C; ++c) gp[size_t(c) * A.p_pad + col] = 0.f;
      }
    }
    fence_before_sync();
  } else {
    // --------------------------------------------- softmax group (warps 6-13)
    const int st = tid - 192;               // 0..255
    const int sw = warp - 6;                // 0..7
    const uint32_t rb_local = smem_u32(rbuf);
    auto label = [&](int64_t u) {           // of the row that this thread owns in tile u
      const int64_t grow = (W.tile0 + u * W.tstride) * kRows + int(rank) * RS + st;
      return u < T && st < RS && grow < A.n ? __ldg(A.y + grow) : -1;
    };
    int ynext = label(0);
    for (int64_t u = 0; u < T && !*abort_flag; ++u) {
      const int slot = int(u % SLOTS);
      const uint32_t use_par = uint32_t((u / SLOTS) & 1);
      if (st == 0) mbar_arrive_expect_tx(&zrdy[slot], uint32_t(kRows) * N * 4);
      if (st < RS) ylab[st] = ynext;
      ynext = label(u + 1);                 // a tile ahead of its use
      // One thread waits for the partials; after the group barrier every thread
      // takes its own cluster-scope acquire of the completed phase.
      const bool zok = (st == 0) ? wait_bounded(&zrdy[slot], use_par, A.spin_limit, abort_flag, true) : true;
      if (!named_bar_soft_and(zok)) {
        if (!zok) fail(ERR_TIMEOUT_EXCHANGE);
        break;
      }
      (void)mbar_test_cluster(smem_u32(&zrdy[slot]), use_par);
      // Softmax with the zero logit of class K, residual and row log-likelihood: four
      // lanes per (owned row, chain), lane q takes the classes q, q + 4, ...; the S
      // partials are summed in rank order, the exponentials pairwise (classes 16, 8, 4,
      // 2 and 1 apart).  With one warp per (row, chain) and a lane per class, 64 rows
      // took 9600 clocks, longer than the MMAs of a tile of 800 columns.
      const float* zsl = zx + size_t(slot) * S * RS * N;
      const uint32_t zsl_s = smem_u32(zsl);
      const int q = st & 3;
      for (int it0 = 0; it0 < RS * chains; it0 += kSoftThreads / 4) {
        const int it = it0 + (st >> 2);
        const bool act = it < RS * chains;
        int il = act ? it : 0, ch = 0;
        if (chains > 1) {
          ch = il / chains;                 // quotient: the row
          const int row = ch;
          ch = il - row * chains;
          il = row;
        }
        const int cb = ch * Km1;
        const int yi = act ? ylab[il] : -1;
        const int zsw = zx_swizzle(il, N);
        float z[8], e[8];
        float mx = zl ? 0.f : -INFINITY;
        uint32_t za[8];                     // of this lane's classes; the last class again where there is none
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          z[j] = 0.f;
          const int el = cb + min(q + 4 * j, Km1 - 1);
          za[j] = zsl_s + uint32_t(il * N * 4 + (((el >> 2) ^ zsw) << 4) + (el & 3) * 4);
        }
        for (int pr = 0; pr < S; ++pr) {
          const uint32_t po = uint32_t(pr * RS * N * 4);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (4 * j >= Km1) continue;
            float t;
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(t) : "r"(za[j] + po));
            z[j] += t;
          }
        }
        // With the zero logit of class K the row maximum includes 0 and the sum
        // e^{-m}; without it (unconstrained layout) only the Km1 free logits count.
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (q + 4 * j < Km1) mx = fmaxf(mx, z[j]);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        float zy = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          e[j] = 0.f;
          if (4 * j >= Km1) continue;
          if (q + 4 * j < Km1) e[j] = expf(z[j] - mx);
          if (j == (yi >> 2)) zy = z[j];
        }
        float se = ((e[0] + e[4]) + (e[2] + e[6])) + ((e[1] + e[5]) + (e[3] + e[7]));
        se += __shfl_xor_sync(0xffffffffu, se, 2);
        se += __shfl_xor_sync(0xffffffffu, se, 1);
        if (zl) se += expf(-mx);
        const bool valid = yi >= 0;
        zy = __shfl_sync(0xffffffffu, zy, (lane & 28) + (yi & 3));
        __nv_bfloat16* rrow = rloc + il * NP;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (4 * j >= Km1) continue;
          const int cls = q + 4 * j, el = cb + cls;
          if (act && cls < Km1)
            rrow[(el & ~63) + ((((el >> 3) & 7) ^ (il & 7)) << 3) + (el & 7)] =
                __float2bfloat16_rn(valid ? ((cls == yi ? 1.f : 0.f) - e[j] / se) : 0.f);
        }
        if (act && q == 0 && valid)
          lacc[il * chains + ch] += double((yi < Km1 ? zy : 0.f) - mx - logf(se));
      }
      // The partials of tile u are consumed: peers may push tile u + 1.
      named_bar_soft();
      if (sw == 1 && lane < S)
        mbar_arrive_remote(S > 1 ? map_peer(smem_u32(&zxfree[slot]), uint32_t(lane)) : smem_u32(&zxfree[slot]));
      // R buffer b = u % rbufs: every CTA's gradient sweep of tile u - rbufs
      // must be done reading it.
      const int rbi = int(u % RBUFS);
      bool fok = true;
      if (u >= RBUFS && st == 0) {
        fok = wait_bounded(&rfreec[rbi], uint32_t(((u - RBUFS) / RBUFS) & 1), A.spin_limit, abort_flag, true);
        if (!fok) fail(ERR_TIMEOUT_EXCHANGE);
      }
      if (!named_bar_soft_and(fok && !*abort_flag)) break;
      // Push the owned R rows into every peer's operand buffer (MN-major,
      // 128-byte swizzle: 16-byte chunk j of row r sits at chunk j ^ (r % 8)).
      for (int it = st; it < RS * C8 * S; it += kSoftThreads) {
        const int peer = it % S, rest = it / S;
        const int c8 = rest % C8, il = rest / C8;
        const int r = int(rank) * RS + il;
        uint4 v;
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "r"(smem_u32(rloc + il * NP + (c8 & ~7) * 8 + (((c8 & 7) ^ (il & 7)) << 3))));
        const uint32_t off = uint32_t((c8 >> 3) * kBoxBytes + r * 128 + (((c8 & 7) ^ (r & 7)) << 4));
        const uint32_t la = rb_local + uint32_t(rbi * rbuf_bytes) + off;
        const uint32_t ra = (S > 1) ? map_peer(la, uint32_t(peer)) : la;
        const uint32_t rbar = (S > 1) ? map_peer(smem_u32(&rfull[rbi]), uint32_t(peer)) : smem_u32(&rfull[rbi]);
        st_async_v4f(ra, __uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w), rbar);
      }
    }
    named_bar_soft();
    if (sw == 0)
      for (int c = lane; c < chains; c += 32) {
        double sum = 0.0;
        for (int il = 0; il < RS; ++il) sum += lacc[il * chains + c];
        A.lpart[(size_t(W.slot) * S + rank) * A.lpart_cstride + c] = sum;
      }
  }
  __syncthreads();
  if (!base && warp == 1) {
    fence_after_sync();
    tmem_dealloc(tmem, A.tmem_cols);
  }
  if (*abort_flag && tid < S) {
    const uint32_t a = smem_u32(stop);
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(S > 1 ? map_peer(a, uint32_t(tid)) : a), "r"(1) : "memory");
  }
  if (S > 1) cluster_sync_all();
  else __syncthreads();
  if (*reinterpret_cast<volatile int*>(stop)) {
    // Without an abort every push between CTAs has been waited for.  After one, some of
    // those that the cluster issued before the barrier may be on their way: the shared
    // memory and the barriers that they go to stay until they have landed.
    __nanosleep(200000);
  } else if (base) {   // the next share lays out its own barriers here
    for (int i = tid; i < 3 * nslots + 6 * kMaxDepth + kMaxAhead + 1 + 4; i += kThreads)
      asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bars + i)) : "memory");
  }
}

template <bool kFP8>
__global__ void __launch_bounds__(kFP8 ? kThreadsFp8 : kThreadsBf16, 1) lpg_tc_kernel(const TcArgs A) {
  const int cl = int(blockIdx.x) / A.S;
  const int64_t nclu = A.nclusters;
  const TcShare W{cl, nclu, cl >= A.ntiles ? 0 : (A.ntiles - 1 - cl) / nclu + 1, cl};
  tc_body<kFP8>(A, W, nullptr, nullptr);
}

// Several independent problems in one launch: cluster k of the grid works off the
// items [first[k], first[k + 1]), each a run of row tiles of one problem with its
// own arguments (X, labels, operand boxes, tile plan, partial slots); every problem
// shares the cluster size and the storage type.  `chains` is the call's chain
// count.  TMEM is taken once for all items.
template <bool kFP8>
__global__ void __launch_bounds__(kFP8 ? kThreadsFp8 : kThreadsBf16, 1)
    lpg_tc_kernel_batched(const TcArgs* __restrict__ table, const TcItem* __restrict__ items,
                          const int* __restrict__ first, int chains) {
  __shared__ TcArgs args;
  __shared__ TcShare share;
  __shared__ uint32_t tbase;
  __shared__ int stop;
  const int k = int(blockIdx.x) / table[0].S;
  const int i1 = first[k + 1];
  if (threadIdx.x == 0) stop = 0;
  if (threadIdx.x / 32 == 1) tmem_alloc(&tbase, 512);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  for (int i = first[k]; i < i1; ++i) {
    if (threadIdx.x == 0) {
      const TcItem it = items[i];
      args = table[it.prob];
      args.chains = chains;
      args.C = chains * args.Km1;
      share = TcShare{it.tile0, 1, it.tiles, it.slot};
    }
    __syncthreads();
    tc_body<kFP8>(args, share, &tbase, &stop);
    __syncthreads();
    if (stop) break;   // the same in every CTA of the cluster (raised before its last barrier)
  }
  if (threadIdx.x / 32 == 1) {
    fence_after_sync();
    tmem_dealloc(tbase, 512);
  }
}

// Coefficients of every problem of a batch into their operand boxes: block
// row b (blockIdx.y) converts problem b.
struct BetaTiles {
  const float* beta;
  const float* scales;
  __nv_bfloat16* out;
  int32_t Km1, N, p_pad;
};

// Byte offset of element (row r, column c) of a 128-byte-swizzled box whose
// rows hold 64 BF16 values: 16-byte chunk (c / 8) is stored at chunk
// (c / 8) ^ (r % 8).
__host__ __device__ inline uint32_t sw128_offset(int r, int c) {
  return uint32_t(r) * 128u + uint32_t(((c >> 3) ^ (r & 7)) << 4) + uint32_t((c & 7) * 2);
}

// X (row-major n x p, float or double) -> BF16 boxes of 128 rows x 64 columns
// in their shared-memory image, [n_pad / 128][p_pad / 64][16 KB]; padding zero.
template <typename IT>
__global__ void x_to_tiles_kernel(const IT* X, __nv_bfloat16* out, int64_t n, int32_t p, int32_t p_pad, int64_t n_pad,
                                  int* err) {
  const int64_t total = n_pad * p_pad;
  const int64_t nkb = p_pad / kBox;
  int bad = 0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t row = i / p_pad, col = i - row * p_pad;
    float v = 0.f;
    if (row < n && col < p) {
      const IT x = X[row * p + col];
      if (!isfinite(double(x))) bad = 1;
      v = float(x);
    }
    const int64_t t = row / kRows, kb = col / kBox;
    const size_t off = size_t(t * nkb + kb) * kBoxBytes + sw128_offset(int(row % kRows), int(col % kBox));
    *reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<unsigned char*>(out) + off) = __float2bfloat16_rn(v);
  }
  if (bad) atomicOr(err, ERR_NONFINITE_X);
}

// X (row-major n x p, float or double) -> FP8 E4M3 boxes of 128 rows x 64
// columns, row-major inside a box, [n_pad / 128][p_pad / 64][8 KB]: x_q =
// RNE-satfinite(x / s_j), the per-column scale s_j computed beforehand.
template <typename IT>
__global__ void x_to_tiles_fp8_kernel(const IT* X, const float* scales, unsigned char* out, int64_t n, int32_t p,
                                      int32_t p_pad, int64_t n_pad, int* err) {
  const int64_t total = n_pad * p_pad;
  const int64_t nkb = p_pad / kBox;
  int bad = 0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t row = i / p_pad, col = i - row * p_pad;
    unsigned char q = 0;
    if (row < n && col < p) {
      const IT x = X[row * p + col];
      if (!isfinite(double(x))) bad = 1;
      q = static_cast<unsigned char>(__nv_cvt_float_to_fp8(float(x) / scales[col], __NV_SATFINITE, __NV_E4M3));
    }
    const int64_t t = row / kRows, kb = col / kBox;
    out[size_t(t * nkb + kb) * kFp8BoxBytes + size_t(row % kRows) * 64 + size_t(col % kBox)] = q;
  }
  if (bad) atomicOr(err, ERR_NONFINITE_X);
}

__global__ void fp8_tiles_to_rows_kernel(const unsigned char* tiles, unsigned char* out, int64_t n, int32_t p,
                                         int32_t p_pad) {
  const int64_t total = n * p;
  const int64_t nkb = p_pad / kBox;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t row = i / p, col = i - row * p;
    const int64_t t = row / kRows, kb = col / kBox;
    out[i] = tiles[size_t(t * nkb + kb) * kFp8BoxBytes + size_t(row % kRows) * 64 + size_t(col % kBox)];
  }
}

// Inverse of x_to_tiles for the stored values (BF16 bits, row-major n x p).
__global__ void tiles_to_rows_kernel(const __nv_bfloat16* tiles, uint16_t* out, int64_t n, int32_t p, int32_t p_pad) {
  const int64_t total = n * p;
  const int64_t nkb = p_pad / kBox;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t row = i / p, col = i - row * p;
    const int64_t t = row / kRows, kb = col / kBox;
    const size_t off = size_t(t * nkb + kb) * kBoxBytes + sw128_offset(int(row % kRows), int(col % kBox));
    out[i] = *reinterpret_cast<const uint16_t*>(reinterpret_cast<const unsigned char*>(tiles) + off);
  }
}

// FP32 coefficients [C][p_pad] -> BF16 operand boxes [p_pad / 64][2N rows x 128 B]
// (hi rows then lo rows; rows C..N-1 of each zero), K-major with the 128-byte
// swizzle.  With FP8 X the column scales are folded in: X B = X_q (diag(s) B).
__global__ void beta_to_tiles_kernel(const float* beta, const float* scales, __nv_bfloat16* out, int C, int N,
                                     int p_pad) {
  const int p8 = p_pad / 8;
  const int64_t total = int64_t(N) * p8;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int k = int(i / p8), col = 8 * int(i - int64_t(k) * p8);
    coef_chunk(beta + size_t(k) * p_pad + col, scales ? scales + col : nullptr, reinterpret_cast<unsigned char*>(out), N, k,
               col, k < C);
  }
}

__global__ void beta_to_tiles_batched_kernel(const BetaTiles* __restrict__ table, int chains) {
  const BetaTiles b = table[blockIdx.y];
  const int C = chains * b.Km1;
  const uint32_t p8 = uint32_t(b.p_pad) / 8, total = uint32_t(b.N) * p8;   // N <= 256
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int k = int(i / p8), col = 8 * int(i - uint32_t(k) * p8);
    coef_chunk(b.beta + size_t(k) * b.p_pad + col, b.scales ? b.scales + col : nullptr,
               reinterpret_cast<unsigned char*>(b.out), b.N, k, col, k < C);
  }
}

}  // namespace tc

// Plan: N = C rounded to 16, MB = PC / 128, TMEM = N * (1 + MB) <= 512.
bool tc_plan(int64_t p, int C, int S, TcPlan* out) {
  const int N = std::max(16, (C + 15) / 16 * 16);
  if (N > 256) return false;
  const int PC = int((p + int64_t(128) * S - 1) / (int64_t(128) * S) * 128);
  const int MB = PC / 128;
  if (N * (1 + MB) > 512) return false;
  // As many logit accumulators as TMEM holds next to the gradient slice.
  const int nz = std::max(1, std::min(kTcMaxDepth, (512 - N * MB) / N));
  const int cols = N * (nz + MB);
  uint32_t tcols = 32;
  while (tcols < uint32_t(cols)) tcols <<= 1;
  out->nz = nz;
  out->slots = out->rbufs = out->la = 1;
  out->N = N;
  out->NP = (N + 63) / 64 * 64;
  out->PC = PC;
  out->MB = MB;
  out->S = S;
  out->tmem_cols = tcols;
  out->stage_bytes = uint32_t(tc::al(size_t(tc::kBoxBytes) + std::max<size_t>(tc::kBoxBytes, size_t(2 * N) * 128), 1024));
  return true;
}

size_t tc_smem_bytes(const TcPlan& pl, int NST, int chains, bool fp8) {
  return tc::smem_layout(NST, pl.stage_bytes, pl.NP, pl.N, pl.S, chains, fp8, pl.slots, pl.rbufs).total;
}

static void (*tc_kernel(bool fp8))(const tc::TcArgs) { return fp8 ? tc::lpg_tc_kernel<true> : tc::lpg_tc_kernel<false>; }
using TcBatchedFn = void (*)(const tc::TcArgs*, const TcItem*, const int*, int);
static TcBatchedFn tc_kernel_batched(bool fp8) {
  return fp8 ? tc::lpg_tc_kernel_batched<true> : tc::lpg_tc_kernel_batched<false>;
}

int tc_threads(bool fp8) { return fp8 ? tc::kThreadsFp8 : tc::kThreadsBf16; }

cudaError_t tc_prepare(size_t smem, int S, bool fp8) {
  cudaError_t e = cudaFuncSetAttribute(tc_kernel(fp8), cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  if (S > 8) e = cudaFuncSetAttribute(tc_kernel(fp8), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

cudaError_t tc_max_active_clusters(size_t smem, int S, bool fp8, int* out) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(S, 1, 1);
  cfg.blockDim = dim3(tc_threads(fp8), 1, 1);
  cfg.dynamicSmemBytes = smem;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(out, tc_kernel(fp8), &cfg);
}

cudaError_t tc_x_to_tiles(int in_dtype, const void* X, void* out, int64_t n, int32_t p, int32_t p_pad, int* err,
                          cudaStream_t s) {
  const int64_t n_pad = (n + tc::kRows - 1) / tc::kRows * tc::kRows;
  const int g = std::max(1, int(std::min<int64_t>(8192, (n_pad * p_pad + 255) / 256)));
  if (in_dtype == HMC_F64)
    tc::x_to_tiles_kernel<double><<<g, 256, 0, s>>>(static_cast<const double*>(X), static_cast<__nv_bfloat16*>(out), n,
                                                    p, p_pad, n_pad, err);
  else
    tc::x_to_tiles_kernel<float><<<g, 256, 0, s>>>(static_cast<const float*>(X), static_cast<__nv_bfloat16*>(out), n,
                                                   p, p_pad, n_pad, err);
  return cudaGetLastError();
}

cudaError_t tc_x_to_tiles_fp8(int in_dtype, const void* X, const float* scales, void* out, int64_t n, int32_t p,
                              int32_t p_pad, int* err, cudaStream_t s) {
  const int64_t n_pad = (n + tc::kRows - 1) / tc::kRows * tc::kRows;
  const int g = std::max(1, int(std::min<int64_t>(8192, (n_pad * p_pad + 255) / 256)));
  if (in_dtype == HMC_F64)
    tc::x_to_tiles_fp8_kernel<double><<<g, 256, 0, s>>>(static_cast<const double*>(X), scales,
                                                        static_cast<unsigned char*>(out), n, p, p_pad, n_pad, err);
  else
    tc::x_to_tiles_fp8_kernel<float><<<g, 256, 0, s>>>(static_cast<const float*>(X), scales,
                                                       static_cast<unsigned char*>(out), n, p, p_pad, n_pad, err);
  return cudaGetLastError();
}

cudaError_t tc_tiles_to_rows(const void* tiles, void* out_bits, int64_t n, int32_t p, int32_t p_pad, bool fp8,
                             cudaStream_t s) {
  const int g = std::max(1, int(std::min<int64_t>(8192, (n * p + 255) / 256)));
  if (fp8)
    tc::fp8_tiles_to_rows_kernel<<<g, 256, 0, s>>>(static_cast<const unsigned char*>(tiles),
                                                   static_cast<unsigned char*>(out_bits), n, p, p_pad);
  else
    tc::tiles_to_rows_kernel<<<g, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(tiles),
                                              static_cast<uint16_t*>(out_bits), n, p, p_pad);
  return cudaGetLastError();
}

cudaError_t tc_beta_to_tiles(const float* beta, const float* scales, void* out, int C, int N, int p_pad,
                             cudaStream_t s) {
  const int64_t total = int64_t(N) * (p_pad / 8);
  const int g = std::max(1, int(std::min<int64_t>(4096, (total + 255) / 256)));
  tc::beta_to_tiles_kernel<<<g, 256, 0, s>>>(beta, scales, static_cast<__nv_bfloat16*>(out), C, N, p_pad);
  return cudaGetLastError();
}

static tc::TcArgs make_args(const TcPlan& pl, const TcLaunch& L) {
  tc::TcArgs a{};
  a.xs = L.xs;
  a.xscale = L.xscale;
  a.fp8 = L.fp8;
  a.bs = static_cast<const __nv_bfloat16*>(L.bs);
  a.n = L.n;
  a.p_pad = L.p_pad;
  a.PC = pl.PC;
  a.S = pl.S;
  a.N = pl.N;
  a.NP = pl.NP;
  a.C = L.C;
  a.Km1 = L.Km1;
  a.chains = L.chains;
  a.MB = pl.MB;
  a.NST = L.NST;
  a.nclusters = L.nclusters;
  a.ntiles = (L.n + tc::kRows - 1) / tc::kRows;
  a.tmem_cols = pl.tmem_cols;
  a.stage_bytes = pl.stage_bytes;
  a.gpart = static_cast<float*>(L.gpart);
  a.gpart_cstride = L.gpart_cstride;
  a.lpart = L.lpart;
  a.lpart_cstride = L.lpart_cstride;
  a.y = L.y;
  a.err = L.err;
  a.spin_limit = L.spin_limit;
  a.inject_timeout = L.inject_timeout;
  a.zlogit = L.zlogit;
  a.nz = pl.nz;
  a.slots = pl.slots;
  a.rbufs = pl.rbufs;
  a.la = pl.la;
  return a;
}

static void tc_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int clusters, int S, bool fp8, size_t smem,
                      cudaStream_t stream) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3(clusters * S, 1, 1);
  cfg.blockDim = dim3(tc_threads(fp8), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

cudaError_t tc_launch(const TcPlan& pl, const TcLaunch& L, size_t smem, cudaStream_t stream) {
  const tc::TcArgs a = make_args(pl, L);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  tc_config(cfg, attr, L.nclusters, pl.S, L.fp8 != 0, smem, stream);
  return cudaLaunchKernelEx(&cfg, tc_kernel(L.fp8 != 0), a);
}

// ---- one launch for several problems
cudaError_t tc_prepare_batched(size_t smem, int S, bool fp8) {
  cudaError_t e = cudaFuncSetAttribute(tc_kernel_batched(fp8), cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  if (S > 8) e = cudaFuncSetAttribute(tc_kernel_batched(fp8), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

cudaError_t tc_max_active_clusters_batched(size_t smem, int S, bool fp8, int* out) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  tc_config(cfg, attr, 1, S, fp8, smem, nullptr);
  return cudaOccupancyMaxActiveClusters(out, tc_kernel_batched(fp8), &cfg);
}

cudaError_t tc_upload_batch(const TcPlan* plans, const TcLaunch* launches, int m, void** d_table) {
  std::vector<tc::TcArgs> t(m);
  for (int b = 0; b < m; ++b) t[b] = make_args(plans[b], launches[b]);
  cudaError_t e = cudaMalloc(d_table, size_t(m) * sizeof(tc::TcArgs));
  if (e != cudaSuccess) return e;
  return cudaMemcpy(*d_table, t.data(), size_t(m) * sizeof(tc::TcArgs), cudaMemcpyHostToDevice);
}

cudaError_t tc_upload_beta_table(const TcBetaBox* boxes, int m, void** d_table) {
  std::vector<tc::BetaTiles> t(m);
  for (int b = 0; b < m; ++b)
    t[b] = tc::BetaTiles{boxes[b].beta, boxes[b].scales, static_cast<__nv_bfloat16*>(boxes[b].out), boxes[b].Km1,
                         boxes[b].N, boxes[b].p_pad};
  cudaError_t e = cudaMalloc(d_table, size_t(m) * sizeof(tc::BetaTiles));
  if (e != cudaSuccess) return e;
  return cudaMemcpy(*d_table, t.data(), size_t(m) * sizeof(tc::BetaTiles), cudaMemcpyHostToDevice);
}

int tc_beta_job_bytes() { return int(sizeof(tc::BetaTiles)); }

cudaError_t tc_beta_to_tiles_batched(const void* d_table, int m, int chains, int64_t max_elems, cudaStream_t s) {
  const int gx = std::max(1, int(std::min<int64_t>(512, (max_elems / 8 + 255) / 256)));
  tc::beta_to_tiles_batched_kernel<<<dim3(gx, m), 256, 0, s>>>(static_cast<const tc::BetaTiles*>(d_table), chains);
  return cudaGetLastError();
}

// Items for `clusters` clusters: the problems' tiles in order, cut so that every
// cluster gets about the same cost.  In units of 1000 clocks, measured per item of 32
// uneven problems: a tile with two tiles of lookahead costs its boxes per CTA, at least
// the exchange (7.6); with one tile of lookahead 4.6 and 0.82 per box; 1.15 times that
// with more than 16 columns; an item's start and the drain of its gradient slice 10.
// The smallest budget per cluster that needs no more clusters is found by bisection;
// max_slots[b] bounds the items of problem b.
// (One cluster at least per problem, by rounded shares, gave 47 clusters to the 35-38
// that fit at once: 32 uneven problems waited for a second wave, 1060 us.)
int tc_make_items(const TcPlan* plans, const int64_t* ntiles, const int* max_slots, int m, int clusters,
                  std::vector<TcItem>* items, std::vector<int>* first, std::vector<int>* slots) {
  const double kItem = 10.0;
  auto cost = [&](int b) {
    const double boxes = plans[b].PC / 64.0;
    return (plans[b].la > 1 ? std::max(7.6, boxes) : 4.6 + 0.82 * boxes) * (plans[b].N > 16 ? 1.15 : 1.0);
  };
  auto build = [&](double budget) {
    items->clear();
    first->assign(1, 0);
    slots->assign(m, 0);
    double left = budget;
    for (int b = 0; b < m; ++b) {
      const double w = cost(b);
      int64_t t = 0;
      while (t < ntiles[b]) {
        int64_t take = int64_t((left - kItem) / w);
        if (take < 1 && left < budget) {   // close this cluster
          first->push_back(int(items->size()));
          left = budget;
          continue;
        }
        take = std::max<int64_t>(1, std::min(take, ntiles[b] - t));
        items->push_back(TcItem{t, int32_t(take), int32_t(b), (*slots)[b]});
        (*slots)[b] += 1;
        t += take;
        left -= kItem + double(take) * w;
      }
    }
    first->push_back(int(items->size()));
    if (int(first->size()) - 1 > clusters) return false;
    for (int b = 0; b < m; ++b)
      if ((*slots)[b] > max_slots[b]) return false;
    return true;
  };
  double lo = 0.0, hi = kItem;
  for (int b = 0; b < m; ++b) hi += kItem + double(ntiles[b]) * cost(b);
  for (int it = 0; it < 60 && hi - lo > 1e-3 * hi; ++it) {
    const double mid = 0.5 * (lo + hi);
    (build(mid) ? hi : lo) = mid;
  }
  build(hi);   // one cluster could hold everything: always feasible
  return int(first->size()) - 1;
}

cudaError_t tc_launch_batched(const void* d_table, const TcItem* d_items, const int* d_first, int chains,
                              int total_clusters, int S, bool fp8, size_t smem, cudaStream_t stream) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  tc_config(cfg, attr, total_clusters, S, fp8, smem, stream);
  return cudaLaunchKernelEx(&cfg, tc_kernel_batched(fp8), static_cast<const tc::TcArgs*>(d_table), d_items, d_first,
                            chains);
}

}  // namespace hmc
