// Per-coefficient kernels of the sampler: fixed-order reduction of the fused
// pass's partial gradients plus the prior term (Eq. gradient), the leapfrog
// momentum / coefficient updates (Eqs. hmc1-hmc3), the momentum draw, the
// Metropolis test with momentum (Eq. accept, kinetic energy eta.eta/2), the
// keep-or-restore select, and the upload / layout conversions.
//
// Scalars (log K, kinetic energy) are summed in FP64: per-block partials in
// fixed slots, combined by the last block of each chain (ticket counter) in a
// fixed tree, so results are bitwise repeatable.
#include <cmath>

#include "device_common.cuh"
#include "internal.h"

namespace hmc {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float prior_term32(float b, int kind, float s) {
  const float x = b / s;
  return kind == HMC_PRIOR_CAUCHY ? -log1pf(x * x) : -0.5f * x * x;
}

// Log-prior term of one coefficient, formed in the state's precision (FP64
// arithmetic is scarce on this GPU) and returned for FP64 accumulation.
template <typename ST>
__device__ __forceinline__ double prior_term(ST b, int kind, double s) {
  if constexpr (sizeof(ST) == 4) {
    return double(prior_term32(float(b), kind, float(s)));
  } else {
    const double x = double(b);
    if (kind == HMC_PRIOR_CAUCHY) return -log1p((x / s) * (x / s));
    return -(x * x) / (2.0 * s * s);
  }
}

// The FP32 prior terms of four coefficients as one FP64 value: summed in FP32 with the
// rounding errors and theirs carried along (Knuth's two-sum, twice; what is dropped is
// 2^-72 of the sum), so that FP64 units see three conversions and two additions, not
// four of each, and round twice.
__device__ __forceinline__ double prior_quad(const float4 b, int kind, float sc) {
  auto term = [&](int i) { return prior_term32(i == 0 ? b.x : i == 1 ? b.y : i == 2 ? b.z : b.w, kind, sc); };
  float t[4] = {term(0), term(1), term(2), term(3)};
  float s = t[0], e = 0.f, e2 = 0.f;
#pragma unroll
  for (int i = 1; i < 4; ++i) {
    s = two_sum(s, t[i], t[i]);
    e = two_sum(e, t[i], t[i]);
    e2 = __fadd_rn(e2, t[i]);
  }
  if (!isfinite(s)) return ((double(term(0)) + double(term(1))) + double(term(2))) + double(term(3));
  return (double(s) + double(e)) + double(e2);
}

template <typename ST>
__device__ __forceinline__ ST prior_deriv(ST b, int kind, double s) {
  if (kind == HMC_PRIOR_CAUCHY) return ST(-2.0) * b / (ST(s * s) + b * b);
  return -b / ST(s * s);
}

// Fixed-order block sums of N doubles: warp 0 sums eight threads' values per lane,
// pairwise, and the lanes in a butterfly; the results are valid in warp 0.  Plain FP64
// additions in a fixed tree: the trees here meet at most a few thousand partials, whose
// rounding stays far below what the accept test or the oracle comparisons can see.  A
// warp's FP64 instruction holds the SM's FP64 units for 16 clocks, so they are few (a
// butterfly in each warp first takes four times as many) and the N sums interleave.
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N]) {
  constexpr int kWarps = kThreads / 32;
  __shared__ double ws[N][kThreads];
  __syncthreads();   // ws may still be read by a previous call
#pragma unroll
  for (int k = 0; k < N; ++k) ws[k][threadIdx.x] = v[k];
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      double t[kWarps];
#pragma unroll
      for (int w = 0; w < kWarps; ++w) t[w] = ws[k][w * 32 + threadIdx.x];
#pragma unroll
      for (int o = kWarps / 2; o > 0; o >>= 1)
#pragma unroll
        for (int w = 0; w < o; ++w) t[w] += t[w + o];
      v[k] = t[0];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < N; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
}

// Thread t's in-order share of v[i * stride], i = t, t + blockDim, ...: four
// interleaved accumulators (fixed assignment, combined in order) keep the
// dependent FP64 chain a quarter as long.
__device__ __forceinline__ double thread_share(const double* v, int n, size_t stride) {
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  int i = threadIdx.x;
  for (; i + 3 * int(blockDim.x) < n; i += 4 * int(blockDim.x)) {
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] += v[size_t(i + u * int(blockDim.x)) * stride];
  }
  for (; i < n; i += blockDim.x) acc[0] += v[size_t(i) * stride];
  return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// Ticket: true in exactly one block (the last to finish) of chain c.
__device__ __forceinline__ bool last_block(unsigned int* ticket, unsigned int nblk) {
  __shared__ int is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = (atomicAdd(ticket, 1u) == nblk - 1u);
  __syncthreads();
  if (is_last) __threadfence();
  return is_last != 0;
}

// Split-K sum of coefficient `idx` over the partials [b0, b1), four loads in flight,
// summed in pairs before they are added: a chain of 22 additions alone cost 3e-8 of the
// gradient (FP32 X, n=6e4 p=785 K=10, 5.6e-8 -> 5.0e-8 in all).  Fours without predicates,
// then the rest: with predicated loads throughout, the reduction of grouped lanes took
// 3 us longer (n=5000 p=3000 K=5, two chains, BF16 X: a leapfrog step of 46.6 us for 43.8).
template <typename ST>
__device__ __forceinline__ ST partial_range_sum(const ST* gpi, int64_t cstride, int b0, int b1) {
  ST g = ST(0);
  int b = b0;
#pragma unroll 2
  for (; b + 4 <= b1; b += 4) {
    ST v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = gpi[size_t(b + k) * cstride];
    g += (v[0] + v[1]) + (v[2] + v[3]);
  }
  if (b < b1) {
    ST v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = b + k < b1 ? gpi[size_t(b + k) * cstride] : ST(0);
    g += (v[0] + v[1]) + v[2];
  }
  return g;
}

// Problem b with first[b] <= block < first[b + 1].
__device__ __forceinline__ int problem_of_block(const int* first, int nprob, int block) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (first[mid] <= block) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// What a call adds to a problem's stored arguments.
template <typename ST>
__device__ __forceinline__ void apply_call(UpdateArgs& A, const UpdateBatch& B, int b) {
  A.chains = B.chains;
  A.eps = B.eps;
  A.temps = B.temps;
  A.thin = B.thin;
  if (B.ugrad) A.ugrad = static_cast<ST*>(B.ugrad) + size_t(B.chains) * B.offset[b];
  if (B.ulogk) A.ulogk = B.ulogk + size_t(b) * B.chains;
}

// The update of coefficient idx (column j of row k = e / p_pad of chain c) from
// its split-K gradient sum g: prior derivative, gradient (also in the user
// layout when asked), momentum and coefficient steps, and the FP64 scalar terms.
template <typename ST>
__device__ __forceinline__ void update_one(const UpdateArgs& A, int mode, int c, int64_t e, int j, size_t idx, ST g,
                                           ST ce, ST eb, double& prior_s, double& kin_s) {
  ST* beta = static_cast<ST*>(A.beta);
  ST* eta = static_cast<ST*>(A.eta);
  ST* grad = static_cast<ST*>(A.grad);
  const ST bv = beta[idx];
  g += prior_deriv(bv, A.prior_kind, A.prior_scale);
  grad[idx] = g;
  if (A.ugrad) {
    ST* ug = static_cast<ST*>(A.ugrad) + size_t(c) * A.ku * A.p;
    const int k = int(e / A.p_pad);
    ug[size_t(k) * A.p + j] = g;
    if (k == 0 && A.ku > A.Km1) ug[size_t(A.Km1) * A.p + j] = ST(0);   // masked row K
  }
  ST ev = ST(0);
  if (mode & (UPD_ETA_HALF | UPD_ETA_FULL)) {
    ev = eta[idx] + ce * g;
    eta[idx] = ev;
  }
  if (mode & UPD_SCALARS) {
    prior_s += prior_term(bv, A.prior_kind, A.prior_scale);
    if (mode & UPD_ACCEPT) kin_s += double(ev) * double(ev);
  }
  if (mode & UPD_BETA) beta[idx] = bv + eb * ev;
}

// GRP: a group of G lanes (A.glanes, a power of two <= 32) shares each coefficient:
// lane l of the group sums the partials [l nparts / G, (l + 1) nparts / G) in
// order and the G range sums meet in a butterfly (every lane of the group ends
// with the same bits: each step adds the same two values); lane 0 of the group
// applies the update.  G = 1 is the plain in-order sum.  V4 (FP32, G = 1, p_pad,
// the slice stride and the state buffers 16-byte aligned): each thread takes four
// consecutive coefficients of one row with 16-byte loads and stores, the same
// arithmetic per coefficient (the gradient sums identical bit for bit); a row's
// last four columns holding padding go through the per-coefficient path.
// What bounds it: latency and the FP64 units, not bytes (C = 76, p = 1e4, 9 slices,
// 28 MB: FP64 pipe 48% busy, 25 us).  With prior_quad, block_sum's few FP64 instructions,
// one sum instead of two where the kinetic energy is not asked for, 32-bit remainders,
// the state loaded before the slices and five blocks on an SM: 17 us; C = 72, p = 2e4:
// 31 -> 24 us; 64 chains of C = 9, p = 2000: 17.6 -> 15.5 us.
// Block bx of the nbx blocks that share chain c.
template <typename ST, bool GRP, bool V4>
__device__ __forceinline__ void reduce_update_body(const UpdateArgs& A, const int mode, const int c, const int bx,
                                                   const int nbx) {
  const int64_t per_chain = int64_t(A.Km1) * A.p_pad;
  const size_t base = size_t(c) * per_chain;
  const ST* gp = static_cast<const ST*>(A.gpart);
  ST* beta = static_cast<ST*>(A.beta);
  ST* eta = static_cast<ST*>(A.eta);
  ST* grad = static_cast<ST*>(A.grad);
  const ST ce = (mode & UPD_ETA_HALF) ? ST(0.5 * A.eps) : ST(A.eps);
  const ST eb = ST(A.eps);
  const int G = GRP ? A.glanes : 1;                 // a power of two
  const int gsh = GRP ? __ffs(G) - 1 : 0;
  const int lane = threadIdx.x & 31, gl = lane & (G - 1);
  const unsigned gmask = G == 32 ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
  const int b0 = (gl * A.nparts) >> gsh, b1 = ((gl + 1) * A.nparts) >> gsh;
  const int64_t stride = (int64_t(nbx) * blockDim.x) >> gsh;
  double prior_s = 0.0, kin_s = 0.0;
  const bool short_rows = per_chain <= 0x7fffffff;   // a 32-bit remainder is a third of a 64-bit one
  auto column = [&](int64_t e) { return short_rows ? int(uint32_t(e) % uint32_t(A.p_pad)) : int(e % A.p_pad); };
  if constexpr (V4) {
    const int64_t n4 = per_chain / 4;
    for (int64_t e4 = int64_t(bx) * blockDim.x + threadIdx.x; e4 < n4; e4 += int64_t(nbx) * blockDim.x) {
      const int64_t e = 4 * e4;
      const int j = column(e);
      if (j >= A.p) continue;  // padding columns stay zero
      const size_t idx = base + size_t(e);
      if (j + 4 > A.p) {
        for (int i = 0; j + i < A.p; ++i)
          update_one<ST>(A, mode, c, e + i, j + i, idx + i, partial_range_sum(gp + idx + i, A.gpart_cstride, 0, A.nparts),
                         ce, eb, prior_s, kin_s);
        continue;
      }
      // Split-K sums of the four coefficients, as partial_range_sum forms them.
      const float4 bv = *reinterpret_cast<const float4*>(beta + idx);
      float4 e0 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (mode & (UPD_ETA_HALF | UPD_ETA_FULL)) e0 = *reinterpret_cast<const float4*>(eta + idx);
      float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
      auto slice = [&](int b) { return *reinterpret_cast<const float4*>(gp + idx + size_t(b) * A.gpart_cstride); };
      auto add4 = [&](const float4& a, const float4& b, const float4& c, const float4& d) {
        g.x += (a.x + b.x) + (c.x + d.x);
        g.y += (a.y + b.y) + (c.y + d.y);
        g.z += (a.z + b.z) + (c.z + d.z);
        g.w += (a.w + b.w) + (c.w + d.w);
      };
      int b = 0;
      for (; b + 4 <= A.nparts; b += 4) add4(slice(b), slice(b + 1), slice(b + 2), slice(b + 3));
      if (b < A.nparts) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        add4(slice(b), b + 1 < A.nparts ? slice(b + 1) : zero, b + 2 < A.nparts ? slice(b + 2) : zero, zero);
      }
      float4 gg;
      gg.x = g.x + prior_deriv(bv.x, A.prior_kind, A.prior_scale);
      gg.y = g.y + prior_deriv(bv.y, A.prior_kind, A.prior_scale);
      gg.z = g.z + prior_deriv(bv.z, A.prior_kind, A.prior_scale);
      gg.w = g.w + prior_deriv(bv.w, A.prior_kind, A.prior_scale);
      *reinterpret_cast<float4*>(grad + idx) = gg;
      if (A.ugrad) {
        ST* ug = static_cast<ST*>(A.ugrad) + size_t(c) * A.ku * A.p;
        const int k = int(e / A.p_pad);
        ST* row = ug + size_t(k) * A.p + j;
        row[0] = gg.x;
        row[1] = gg.y;
        row[2] = gg.z;
        row[3] = gg.w;
        if (k == 0 && A.ku > A.Km1)   // masked row K
          for (int i = 0; i < 4; ++i) ug[size_t(A.Km1) * A.p + j + i] = ST(0);
      }
      float4 ev = make_float4(0.f, 0.f, 0.f, 0.f);
      if (mode & (UPD_ETA_HALF | UPD_ETA_FULL)) {
        ev = make_float4(e0.x + ce * gg.x, e0.y + ce * gg.y, e0.z + ce * gg.z, e0.w + ce * gg.w);
        *reinterpret_cast<float4*>(eta + idx) = ev;
      }
      if (mode & UPD_SCALARS) {
        prior_s += prior_quad(bv, A.prior_kind, float(A.prior_scale));
        if (mode & UPD_ACCEPT)
          kin_s += ((double(ev.x) * double(ev.x) + double(ev.y) * double(ev.y)) + double(ev.z) * double(ev.z)) +
                   double(ev.w) * double(ev.w);
      }
      if (mode & UPD_BETA)
        *reinterpret_cast<float4*>(beta + idx) =
            make_float4(bv.x + eb * ev.x, bv.y + eb * ev.y, bv.z + eb * ev.z, bv.w + eb * ev.w);
    }
  } else {
    for (int64_t e = (int64_t(bx) * blockDim.x + threadIdx.x) >> gsh; e < per_chain; e += stride) {
      const int j = column(e);
      if (j >= A.p) continue;  // padding columns stay zero (the whole group skips)
      const size_t idx = base + size_t(e);
      ST g = partial_range_sum(gp + idx, A.gpart_cstride, b0, b1);
      if (GRP) {
        for (int o = 1; o < G; o <<= 1) g += __shfl_xor_sync(gmask, g, o);
        if (gl != 0) continue;
      }
      update_one<ST>(A, mode, c, e, j, idx, g, ce, eb, prior_s, kin_s);
    }
  }
  if (!(mode & UPD_SCALARS)) return;
  double bs[2] = {prior_s, kin_s};
  if (mode & UPD_ACCEPT) {
    block_sum<2>(bs);
  } else {
    double ps[1] = {prior_s};
    block_sum<1>(ps);
    bs[0] = ps[0];
    bs[1] = 0.0;
  }
  if (threadIdx.x == 0) {
    double* sl = A.scal + (size_t(c) * A.nblk + bx) * 2;
    sl[0] = bs[0];
    sl[1] = bs[1];
  }
  if (!last_block(A.tickets + c, unsigned(nbx))) return;
  // The whole last block sums the block partials and the log-likelihood
  // partials of the gradient pass, each in a fixed order, in one tree.
  const double* sl = A.scal + size_t(c) * A.nblk * 2;
  double tot[3] = {thread_share(sl, nbx, 2), thread_share(sl + 1, nbx, 2),
                   thread_share(A.lpart + c, A.nlparts, size_t(A.lpart_cstride))};
  block_sum<3>(tot);
  const double prv = tot[0], kiv = tot[1], liv = tot[2];
  if (threadIdx.x != 0) return;
  const double logk = liv + prv;
  A.tickets[c] = 0u;
  if (!(mode & UPD_ACCEPT)) {
    A.logk[c] = logk;
    if (A.ulogk) A.ulogk[c] = logk;
    return;
  }
  const int64_t it = *A.iter;
  const double T = A.temps ? A.temps[*A.local_iter] : 1.0;
  const double h0 = A.h0[c];
  const double h1 = -logk + 0.5 * kiv;
  const bool finite = isfinite(h1);
  const double u = accept_uniform(*A.seed, uint64_t(it), uint64_t(c) | (uint64_t(A.chains_word_hi) << 32));
  const bool acc = finite && (log(u) < (h0 - h1) / T);
  A.accept[c] = acc ? 1 : 0;
  hmc_chain_stats* st = static_cast<hmc_chain_stats*>(A.stats) + c;
  st->iterations += 1;
  st->accepted += acc ? 1 : 0;
  st->diverged += finite ? 0 : 1;
  if (finite) st->sum_abs_dH += fabs(h1 - h0);
  const double kept = acc ? logk : A.logk0[c];
  A.logk[c] = kept;
  st->logpost = kept;
}

template <typename ST, bool GRP, bool V4>
__global__ void __launch_bounds__(kThreads, V4 ? 5 : 1) reduce_update_kernel(const UpdateArgs A, int mode) {
  chain_wait();
  chain_next();
  reduce_update_body<ST, GRP, V4>(A, mode, int(blockIdx.y), int(blockIdx.x), int(gridDim.x));
}

// The same for every problem of a batch handle in one launch: blocks
// [first[b], first[b + 1]) of grid.x reduce problem b, each problem by the variant
// it takes by itself (so its sums keep their order).  One launch per problem left
// the GPU to 10-20 us kernels of a few blocks each, one after the other: 32 uneven
// problems took 450 us for their reductions, 22 us in one launch.
template <typename ST>
__global__ void __launch_bounds__(kThreads) reduce_update_batched_kernel(const UpdateBatch B, int mode) {
  __shared__ UpdateArgs A;
  __shared__ int sb;
  if (threadIdx.x < 32) {
    const int b = problem_of_block(B.first, B.nprob, int(blockIdx.x));
    const uint32_t* src = reinterpret_cast<const uint32_t*>(B.table + b);
    for (int i = threadIdx.x; i < int(sizeof(UpdateArgs) / 4); i += 32) reinterpret_cast<uint32_t*>(&A)[i] = src[i];
    __syncwarp();
    if (threadIdx.x == 0) {
      sb = b;
      apply_call<ST>(A, B, b);
    }
  }
  __syncthreads();
  const int b = sb, bx = int(blockIdx.x) - B.first[b], nbx = B.first[b + 1] - B.first[b], c = int(blockIdx.y);
  if (A.variant == kUpdGroup)
    reduce_update_body<ST, true, false>(A, mode, c, bx, nbx);
  else if (sizeof(ST) == 4 && A.variant == kUpdVec4)
    reduce_update_body<float, false, true>(A, mode, c, bx, nbx);
  else
    reduce_update_body<ST, false, false>(A, mode, c, bx, nbx);
}

// Start of a trajectory: eta ~ N(0, I), save (beta, grad, log K), H0, then
// the first momentum half step and the first coefficient step.
template <typename ST>
__global__ void __launch_bounds__(kThreads) traj_start_kernel(const UpdateArgs A) {
  const int c = blockIdx.y;
  const int64_t per_chain_q = int64_t(A.Km1) * A.p;
  const int64_t nqb = (per_chain_q + 3) / 4;
  const size_t base = size_t(c) * A.Km1 * A.p_pad;
  ST* beta = static_cast<ST*>(A.beta);
  ST* eta = static_cast<ST*>(A.eta);
  const ST* grad = static_cast<const ST*>(A.grad);
  ST* beta0 = static_cast<ST*>(A.beta0);
  ST* grad0 = static_cast<ST*>(A.grad0);
  const uint64_t it = uint64_t(*A.iter);
  const uint64_t seed = *A.seed;
  const uint64_t chain_word = uint64_t(c) | (uint64_t(A.chains_word_hi) << 32);
  const ST half = ST(0.5 * A.eps), full = ST(A.eps);
  double kin = 0.0;
  for (int64_t qb = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; qb < nqb; qb += int64_t(gridDim.x) * blockDim.x) {
    double z[4];
    momentum_block(seed, it, chain_word, uint64_t(qb), z);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int64_t q = qb * 4 + r;
      if (q >= per_chain_q) break;
      const int64_t k = q / A.p, j = q - k * A.p;
      const size_t idx = base + size_t(k) * A.p_pad + size_t(j);
      const ST e = ST(z[r]);
      kin += double(e) * double(e);
      const ST b = beta[idx], g = grad[idx];
      beta0[idx] = b;
      grad0[idx] = g;
      const ST eh = e + half * g;
      eta[idx] = eh;
      beta[idx] = b + full * eh;
    }
  }
  double kb[1] = {kin};
  block_sum<1>(kb);
  if (threadIdx.x == 0) A.scal[(size_t(c) * A.nblk + blockIdx.x) * 2 + 1] = kb[0];
  if (!last_block(A.tickets + c, gridDim.x)) return;
  double kt[1] = {thread_share(A.scal + size_t(c) * A.nblk * 2 + 1, int(gridDim.x), 2)};
  block_sum<1>(kt);
  const double kiv = kt[0];
  if (threadIdx.x != 0) return;
  A.tickets[c] = 0u;
  A.logk0[c] = A.logk[c];
  A.h0[c] = -A.logk[c] + 0.5 * kiv;
}

// Keep the proposal or restore the trajectory start; write the sample; the
// last block advances the iteration counters.
template <typename ST>
__global__ void __launch_bounds__(kThreads) select_kernel(const UpdateArgs A, unsigned int* ticket_all) {
  const int c = blockIdx.y;
  const int64_t per_chain = int64_t(A.Km1) * A.p_pad;
  const size_t base = size_t(c) * per_chain;
  ST* beta = static_cast<ST*>(A.beta);
  ST* grad = static_cast<ST*>(A.grad);
  const ST* beta0 = static_cast<const ST*>(A.beta0);
  const ST* grad0 = static_cast<const ST*>(A.grad0);
  const bool acc = A.accept[c] != 0;
  const int64_t li = *A.local_iter;
  ST* out = nullptr;
  if (A.samples && ((li + 1) % A.thin) == 0) {
    const int64_t slot = (li + 1) / A.thin - 1;
    out = static_cast<ST*>(A.samples) + size_t(slot) * A.sample_slot_stride + size_t(c) * A.ku * A.p;
    // Rows past the free ones (the masked row K) are zero in every sample.
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < int64_t(A.ku - A.Km1) * A.p;
         e += int64_t(gridDim.x) * blockDim.x)
      out[size_t(A.Km1) * A.p + size_t(e)] = ST(0);
  }
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < per_chain;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t k = e / A.p_pad, j = e - k * A.p_pad;
    if (j >= A.p) continue;
    const size_t idx = base + size_t(e);
    ST b = beta[idx];
    if (!acc) {
      b = beta0[idx];
      beta[idx] = b;
      grad[idx] = grad0[idx];
    }
    if (out) out[size_t(k) * A.p + size_t(j)] = b;
  }
  __shared__ int is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = (atomicAdd(ticket_all, 1u) == gridDim.x * gridDim.y - 1u);
  __syncthreads();
  if (is_last && threadIdx.x == 0) {
    __threadfence();
    *ticket_all = 0u;
    *A.iter += 1;
    *A.local_iter += 1;
  }
}

// Four values of a row, 16 bytes at a time where T is 4 bytes wide.
template <typename T>
struct alignas(16) Quad {
  T v[4];
};
__device__ __forceinline__ bool quad_aligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// hmc_leapfrog start: first half step of the momentum and first coefficient step.
template <typename ST>
__global__ void leap_start_kernel(const UpdateArgs A, int64_t total) {
  ST* beta = static_cast<ST*>(A.beta);
  ST* eta = static_cast<ST*>(A.eta);
  const ST* grad = static_cast<const ST*>(A.grad);
  const ST half = ST(0.5 * A.eps), full = ST(A.eps);
  const int64_t first = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, step = int64_t(gridDim.x) * blockDim.x;
  if (total % 4 == 0 && quad_aligned(beta) && quad_aligned(eta) && quad_aligned(grad)) {
    for (int64_t i = first; i < total / 4; i += step) {
      Quad<ST> b = reinterpret_cast<const Quad<ST>*>(beta)[i], e = reinterpret_cast<const Quad<ST>*>(eta)[i];
      const Quad<ST> g = reinterpret_cast<const Quad<ST>*>(grad)[i];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        e.v[k] = e.v[k] + half * g.v[k];
        b.v[k] = b.v[k] + full * e.v[k];
      }
      reinterpret_cast<Quad<ST>*>(eta)[i] = e;
      reinterpret_cast<Quad<ST>*>(beta)[i] = b;
    }
    return;
  }
  for (int64_t i = first; i < total; i += step) {
    const ST e = eta[i] + half * grad[i];
    eta[i] = e;
    beta[i] = beta[i] + full * e;
  }
}

// Rows of p values (`ku` to a chain, the first km1 of them taken) -> rows of p_pad, the
// rest zero: items first, first + step, ... of this launch.  A quad per item and 32-bit
// indices where they reach: with one value per item and 64-bit remainders 76 rows of
// 10000 took 8.0 us, 576 rows of 2000 10.7 us; now 3.7 and 4.2 us.
template <typename T>
__device__ __forceinline__ void pack_rows(const T* src, T* dst, int64_t chains, int32_t ku, int32_t km1, int32_t p,
                                          int32_t p_pad, int64_t first, int64_t step) {
  const int64_t total = chains * km1 * p_pad;
  if (p_pad % 4 == 0 && total <= 0x7fffffff && quad_aligned(dst)) {
    const uint32_t p4 = uint32_t(p_pad) / 4, n4 = uint32_t(total / 4);
    for (uint32_t i = uint32_t(first); i < n4; i += uint32_t(step)) {
      const uint32_t r = i / p4, c = ku == km1 ? 0u : r / uint32_t(km1);
      const int32_t j = 4 * int32_t(i - r * p4);
      const T* s = src + (size_t(r) + size_t(c) * uint32_t(ku - km1)) * p + j;
      Quad<T> q;
#pragma unroll
      for (int e = 0; e < 4; ++e) q.v[e] = j + e < p ? s[e] : T(0);
      *reinterpret_cast<Quad<T>*>(dst + size_t(i) * 4) = q;
    }
    return;
  }
  for (int64_t i = first; i < total; i += step) {
    const int64_t r = i / p_pad, j = i - r * p_pad;
    const int64_t c = r / km1, k = r - c * km1;
    dst[i] = (j < p) ? src[(c * ku + k) * p + j] : T(0);
  }
}

// [chains][ku][p] -> [chains][km1][p_pad]: rows past km1 of a chain are dropped,
// padding columns are zero.
template <typename T>
__global__ void pack_kernel(const T* src, T* dst, int64_t chains, int32_t ku, int32_t km1, int32_t p, int32_t p_pad) {
  chain_wait();
  chain_next();
  pack_rows(src, dst, chains, ku, km1, p, p_pad, int64_t(blockIdx.x) * blockDim.x + threadIdx.x,
            int64_t(gridDim.x) * blockDim.x);
}

// pack_kernel for every problem of a batch handle in one launch (blocks
// [pfirst[b], pfirst[b + 1]) of grid.x): the problems' blocks of `src` follow one
// another.  `which` picks the coefficients, momenta or gradients.
template <typename T>
__global__ void pack_batched_kernel(const UpdateBatch B, const T* src, int which) {
  const int b = problem_of_block(B.pfirst, B.nprob, int(blockIdx.x));
  const UpdateArgs& A = B.table[b];
  const int32_t ku = A.ku, km1 = A.Km1, p = A.p, p_pad = A.p_pad;
  T* dst = static_cast<T*>(which == 0 ? A.beta : which == 1 ? A.eta : A.grad);
  const T* sp = src + size_t(B.chains) * B.offset[b];
  pack_rows(sp, dst, B.chains, ku, km1, p, p_pad, int64_t(int(blockIdx.x) - B.pfirst[b]) * blockDim.x + threadIdx.x,
            int64_t(B.pfirst[b + 1] - B.pfirst[b]) * blockDim.x);
}

// [chains][km1][p_pad] -> [chains][ku][p]: rows past km1 of a chain are zero.
template <typename T>
__global__ void unpack_kernel(const T* src, T* dst, int64_t chains, int32_t ku, int32_t km1, int32_t p,
                              int32_t p_pad) {
  const int64_t total = chains * ku * p;
  const int64_t first = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, step = int64_t(gridDim.x) * blockDim.x;
  if (total <= 0x7fffffff) {
    const bool quads = p % 4 == 0 && p_pad % 4 == 0 && quad_aligned(src) && quad_aligned(dst);
    const uint32_t w = quads ? uint32_t(p) / 4 : uint32_t(p), n = quads ? uint32_t(total / 4) : uint32_t(total);
    for (uint32_t i = uint32_t(first); i < n; i += uint32_t(step)) {
      const uint32_t r = i / w, j = i - r * w;
      const uint32_t c = ku == km1 ? 0u : r / uint32_t(ku);
      const bool has = ku == km1 || r - c * uint32_t(ku) < uint32_t(km1);
      const T* s = src + (size_t(r) - size_t(c) * uint32_t(ku - km1)) * p_pad;
      if (quads)
        *reinterpret_cast<Quad<T>*>(dst + size_t(i) * 4) = has ? *reinterpret_cast<const Quad<T>*>(s + 4 * j) : Quad<T>{};
      else
        dst[i] = has ? s[j] : T(0);
    }
    return;
  }
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / p, j = i - r * p;
    const int64_t c = r / ku, k = r - c * ku;
    dst[i] = (k < km1) ? src[(c * km1 + k) * p_pad + j] : T(0);
  }
}

template <typename IT>
__device__ __forceinline__ float to_f32(IT v) {
  return float(v);
}

template <typename IT, typename XT>
__global__ void convert_x_kernel(const IT* src, XT* dst, const float* scales, int64_t n, int32_t p, int32_t p_pad,
                                 int* err) {
  const int64_t total = n * p_pad;
  int bad = 0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / p_pad, j = i - r * p_pad;
    if (j >= p) {
      dst[i] = XT(0.0f);
      continue;
    }
    const IT v = src[r * p + j];
    if (!isfinite(double(v))) bad = 1;
    if constexpr (std::is_same<XT, double>::value) {
      dst[i] = double(v);
    } else if constexpr (std::is_same<XT, float>::value) {
      dst[i] = float(v);
    } else if constexpr (std::is_same<XT, __nv_bfloat16>::value) {
      dst[i] = __float2bfloat16_rn(float(v));
    } else {
      const float q = float(v) / scales[j];
      __nv_fp8_e4m3 o;
      o.__x = __nv_cvt_float_to_fp8(q, __NV_SATFINITE, __NV_E4M3);
      dst[i] = o;
    }
  }
  if (bad) atomicOr(err, ERR_NONFINITE_X);
}

template <typename IT>
__global__ void fp8_scale_kernel(const IT* src, float* scales, int64_t n, int32_t p, int32_t p_pad) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= p_pad) return;
  if (j >= p) {
    scales[j] = 1.0f;
    return;
  }
  float amax = 0.0f;
  for (int64_t r = 0; r < n; ++r) amax = fmaxf(amax, fabsf(float(src[r * p + j])));
  scales[j] = (amax == 0.0f) ? 1.0f : amax / 448.0f;
}

__global__ void check_labels_kernel(const int32_t* y, int64_t n, int32_t K, int* err) {
  int bad = 0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    if (y[i] < 0 || y[i] >= K) bad = 1;
  if (bad) atomicOr(err, ERR_BAD_LABEL);
}

__global__ void init_stats_kernel(hmc_chain_stats* s, int chains) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < chains) s[c] = hmc_chain_stats{0, 0, 0, 0.0, 0.0};
}

int grid_for(int64_t work, int cap = 4096) {
  int64_t g = (work + kThreads - 1) / kThreads;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return int(g);
}

}  // namespace

int update_group_lanes(int64_t per_chain, int chains, int nparts, int nsm) {
  // Lanes sharing one coefficient's split-K sum: more where few coefficients
  // meet many partials (a small call waits for about nparts / 8 dependent load
  // rounds), while the threads stay within half a wave.
  int G = 1;
  while (G < 32 && nparts >= 16 * G && per_chain * chains * G * 2 <= int64_t(nsm) * 2048) G *= 2;
  return G;
}

int update_blocks_per_chain(int64_t per_chain) {
  // About one coefficient (times its group lanes) per thread: the split-K sum
  // is latency-bound.
  int64_t g = (per_chain + kThreads - 1) / kThreads;
  if (g < 1) g = 1;
  if (g > 1024) g = 1024;
  return int(g);
}

int update_variant(int st, const UpdateArgs& a, int* blocks) {
  auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
  *blocks = a.nblk;
  if (a.glanes > 1) return kUpdGroup;
  if (st == HMC_F64 || a.p_pad % 4 != 0 || a.gpart_cstride % 4 != 0 || !al16(a.gpart) || !al16(a.beta) || !al16(a.eta) ||
      !al16(a.grad))
    return kUpdPlain;
  // four coefficients per thread: a quarter of the blocks (their partial slots and
  // the last-block ticket follow the number of blocks)
  *blocks = std::max(1, (a.nblk + 3) / 4);
  return kUpdVec4;
}

cudaError_t launch_reduce_update(int st, const UpdateArgs& a, int mode, cudaStream_t s) {
  int blocks = 0;
  const int v = update_variant(st, a, &blocks);
  const dim3 grid(blocks, a.chains);
  if (st == HMC_F64) {
    return launch_chained(v == kUpdGroup ? reduce_update_kernel<double, true, false> : reduce_update_kernel<double, false, false>,
                          grid, kThreads, 0, s, a, mode);
  }
  return launch_chained(v == kUpdGroup  ? reduce_update_kernel<float, true, false>
                        : v == kUpdVec4 ? reduce_update_kernel<float, false, true>
                                        : reduce_update_kernel<float, false, false>,
                        grid, kThreads, 0, s, a, mode);
}

cudaError_t launch_reduce_update_batched(int st, const UpdateBatch& b, int mode, cudaStream_t s) {
  const dim3 grid(b.blocks, b.chains);
  if (st == HMC_F64) reduce_update_batched_kernel<double><<<grid, kThreads, 0, s>>>(b, mode);
  else reduce_update_batched_kernel<float><<<grid, kThreads, 0, s>>>(b, mode);
  return cudaGetLastError();
}

int pack_blocks(int64_t elems) { return grid_for((elems + 3) / 4, 1024); }

cudaError_t launch_pack_batched(int st, const UpdateBatch& b, const void* src, int which, cudaStream_t s) {
  if (st == HMC_F64) pack_batched_kernel<double><<<b.pblocks, kThreads, 0, s>>>(b, static_cast<const double*>(src), which);
  else pack_batched_kernel<float><<<b.pblocks, kThreads, 0, s>>>(b, static_cast<const float*>(src), which);
  return cudaGetLastError();
}

cudaError_t launch_traj_start(int st, const UpdateArgs& a, cudaStream_t s) {
  dim3 grid(a.nblk, a.chains);
  if (st == HMC_F64)
    traj_start_kernel<double><<<grid, kThreads, 0, s>>>(a);
  else
    traj_start_kernel<float><<<grid, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_select(int st, const UpdateArgs& a, unsigned int* ticket_all, cudaStream_t s) {
  dim3 grid(a.nblk, a.chains);
  if (st == HMC_F64)
    select_kernel<double><<<grid, kThreads, 0, s>>>(a, ticket_all);
  else
    select_kernel<float><<<grid, kThreads, 0, s>>>(a, ticket_all);
  return cudaGetLastError();
}

cudaError_t launch_leap_start(int st, const UpdateArgs& a, cudaStream_t s) {
  const int64_t total = int64_t(a.chains) * a.Km1 * a.p_pad;
  if (st == HMC_F64)
    leap_start_kernel<double><<<grid_for((total + 3) / 4), kThreads, 0, s>>>(a, total);
  else
    leap_start_kernel<float><<<grid_for((total + 3) / 4), kThreads, 0, s>>>(a, total);
  return cudaGetLastError();
}

cudaError_t launch_pack(int st, const void* src, void* dst, int64_t chains, int32_t ku, int32_t km1, int32_t p,
                        int32_t p_pad, cudaStream_t s) {
  const int g = grid_for((chains * km1 * p_pad + 3) / 4);
  if (st == HMC_F64)
    return launch_chained(pack_kernel<double>, g, kThreads, 0, s, static_cast<const double*>(src),
                          static_cast<double*>(dst), chains, ku, km1, p, p_pad);
  return launch_chained(pack_kernel<float>, g, kThreads, 0, s, static_cast<const float*>(src), static_cast<float*>(dst),
                        chains, ku, km1, p, p_pad);
}

cudaError_t launch_unpack(int st, const void* src, void* dst, int64_t chains, int32_t ku, int32_t km1, int32_t p,
                          int32_t p_pad, cudaStream_t s) {
  const int g = grid_for(chains * ku * p);
  if (st == HMC_F64)
    unpack_kernel<double><<<g, kThreads, 0, s>>>(static_cast<const double*>(src), static_cast<double*>(dst), chains, ku,
                                                 km1, p, p_pad);
  else
    unpack_kernel<float><<<g, kThreads, 0, s>>>(static_cast<const float*>(src), static_cast<float*>(dst), chains, ku,
                                                km1, p, p_pad);
  return cudaGetLastError();
}

template <typename IT>
static cudaError_t convert_from(const IT* src, int xt, void* dst, const float* scales, int64_t n, int32_t p, int32_t p_pad,
                                int* err, cudaStream_t s) {
  const int g = grid_for(n * p_pad, 8192);
  switch (xt) {
    case HMC_F64:
      convert_x_kernel<IT, double><<<g, kThreads, 0, s>>>(src, static_cast<double*>(dst), scales, n, p, p_pad, err);
      break;
    case HMC_F32:
      convert_x_kernel<IT, float><<<g, kThreads, 0, s>>>(src, static_cast<float*>(dst), scales, n, p, p_pad, err);
      break;
    case HMC_BF16:
      convert_x_kernel<IT, __nv_bfloat16><<<g, kThreads, 0, s>>>(src, static_cast<__nv_bfloat16*>(dst), scales, n, p,
                                                                   p_pad, err);
      break;
    default:
      convert_x_kernel<IT, __nv_fp8_e4m3><<<g, kThreads, 0, s>>>(src, static_cast<__nv_fp8_e4m3*>(dst), scales, n, p,
                                                                   p_pad, err);
  }
  return cudaGetLastError();
}

cudaError_t launch_convert_x(int in_dtype, const void* src, int xt, void* dst, const float* scales, int64_t n, int32_t p,
                             int32_t p_pad, int* err, cudaStream_t s) {
  if (in_dtype == HMC_F64) return convert_from(static_cast<const double*>(src), xt, dst, scales, n, p, p_pad, err, s);
  return convert_from(static_cast<const float*>(src), xt, dst, scales, n, p, p_pad, err, s);
}

cudaError_t launch_fp8_scales(int in_dtype, const void* src, float* scales, int64_t n, int32_t p, int32_t p_pad,
                              cudaStream_t s) {
  const int g = (p_pad + kThreads - 1) / kThreads;
  if (in_dtype == HMC_F64)
    fp8_scale_kernel<double><<<g, kThreads, 0, s>>>(static_cast<const double*>(src), scales, n, p, p_pad);
  else
    fp8_scale_kernel<float><<<g, kThreads, 0, s>>>(static_cast<const float*>(src), scales, n, p, p_pad);
  return cudaGetLastError();
}

cudaError_t launch_check_labels(const int32_t* y, int64_t n, int32_t K, int* err, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  check_labels_kernel<<<grid_for(n), kThreads, 0, s>>>(y, n, K, err);
  return cudaGetLastError();
}

cudaError_t launch_init_stats(void* stats, int chains, cudaStream_t s) {
  init_stats_kernel<<<(chains + 127) / 128, 128, 0, s>>>(static_cast<hmc_chain_stats*>(stats), chains);
  return cudaGetLastError();
}

}  // namespace hmc
