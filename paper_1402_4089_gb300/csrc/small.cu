// Small problems on CUDA cores: a gradient, a whole leapfrog trajectory or whole HMC
// iterations of one chain in one launch (Eqs. softmax, loglike, logkernel, gradient,
// hmc1-hmc3 and accept; FP64 or FP32 X and state).
//
// A small gradient is bound by launches and by the latency of passing partial sums
// through global memory: n=1000 p=50 K=3 in FP64 took 20.6 us a leapfrog step as two
// launches and takes 10.6 here (a chain of FP64 operations, about 100 clocks each, most
// of it: dots 5500, softmax 4200, X^T R 7600 of 20700 clocks), n=100 p=10 K=2 in FP32
// 10.2 and 2.3.
// Here a cluster of S CTAs keeps X in shared memory (rows split over the CTAs), every
// CTA holds all coefficients, and a step is
//   logits, softmax and residual of the CTA's rows, its share of X^T R, each
//   coefficient's partial pushed into the shared memory of the CTA that owns the
//   coefficient  -> cluster barrier ->
//   the owner adds the S partials in rank order and the prior, moves momentum and
//   coefficient, and pushes the coefficient into every CTA  -> cluster barrier.
// One cluster per chain; chains run side by side (X is read once per chain, from L2).
// Sums have a fixed order (lanes in a butterfly, CTAs in rank order): repeatable bit
// for bit.  Waits are hardware cluster barriers that every CTA reaches.
#include <algorithm>
#include <cmath>

#include "device_common.cuh"
#include "internal.h"

namespace hmc {
namespace small {

constexpr int kThreads = 512;
constexpr int kCB = 4;          // classes a thread takes together (each X value loaded feeds kCB sums)

template <typename AT>
__device__ __forceinline__ AT ex(AT x);
template <>
__device__ __forceinline__ float ex<float>(float x) { return expf(x); }
template <>
__device__ __forceinline__ double ex<double>(double x) { return exp(x); }
template <typename AT>
__device__ __forceinline__ AT lg(AT x);
template <>
__device__ __forceinline__ float lg<float>(float x) { return logf(x); }
template <>
__device__ __forceinline__ double lg<double>(double x) { return log(x); }

// Prior term and derivative of one coefficient, formed as the reduction kernel forms them.
template <typename ST>
__device__ __forceinline__ double prior_term(ST b, int kind, double s) {
  if constexpr (sizeof(ST) == 4) {
    const float x = float(b) / float(s);
    if (kind == HMC_PRIOR_CAUCHY) return double(-log1pf(x * x));
    return double(-0.5f * x * x);
  } else {
    const double x = double(b);
    if (kind == HMC_PRIOR_CAUCHY) return -log1p((x / s) * (x / s));
    return -(x * x) / (2.0 * s * s);
  }
}
// s2 = s * s.
template <typename ST>
__device__ __forceinline__ ST prior_deriv(ST b, int kind, ST s2) {
  if (kind == HMC_PRIOR_CAUCHY) return ST(-2.0) * b / (s2 + b * b);
  return -b / s2;
}

__device__ __forceinline__ void st_peer(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// a[i] += sum over k = k0, k0 + G, ... < n of x[k * xs] * b[i * bs + k], i < NC.  NC is
// a constant: a predicated multiply of a class past the last would still take its
// turn on the FP64 units.
template <int NC, typename AT>
__device__ __forceinline__ void dots(AT (&a)[kCB], const AT* x, int xs, const AT* b, int bs, int k0, int n, int G) {
#pragma unroll 4
  for (int k = k0; k < n; k += G) {
    const AT v = x[k * xs];
#pragma unroll
    for (int i = 0; i < NC; ++i) a[i] = fma(v, b[i * bs + k], a[i]);
  }
}
template <typename AT>
__device__ __forceinline__ void dots_n(int nc, AT (&a)[kCB], const AT* x, int xs, const AT* b, int bs, int k0, int n,
                                       int G) {
  if (nc == 4) dots<4>(a, x, xs, b, bs, k0, n, G);
  else if (nc == 3) dots<3>(a, x, xs, b, bs, k0, n, G);
  else if (nc == 2) dots<2>(a, x, xs, b, bs, k0, n, G);
  else dots<1>(a, x, xs, b, bs, k0, n, G);
}

struct Layout {
  size_t x, beta, recv, z, rowv, own, scal, total;
  int pitch, rows, own_n;
};
// Coefficients are owned in runs of own_n (a multiple of 4: one block of the momentum draw).
__host__ __device__ inline Layout layout(int64_t n, int p, int C, int S, size_t b) {
  Layout L;
  L.rows = int((n + S - 1) / S);
  L.pitch = p | 1;                       // odd: rows of a column spread over the banks
  const int E = C * p;
  L.own_n = ((E + S - 1) / S + 3) / 4 * 4;
  auto al = [](size_t v) { return (v + 15) & ~size_t(15); };
  size_t off = 0;
  L.scal = off;  off += size_t(16) * 4 * 8 + 64 + size_t(kThreads / 32) * 4 * 8;   // [S][4] sums, decision, warp sums
  L.x = off;     off = al(off + size_t(L.rows) * L.pitch * b);
  L.beta = off;  off = al(off + size_t(S) * L.own_n * b);            // [C][p], then unused
  L.recv = off;  off = al(off + size_t(S) * L.own_n * b);            // [S][own_n] partials received
  L.z = off;     off = al(off + size_t(L.rows) * C * b);             // [C][rows] logits, then residuals
  L.rowv = off;  off = al(off + size_t(L.rows) * (2 * b + 4));       // per row: maximum, then 1 / sum; e^-m; label
  L.own = off;   off = al(off + size_t(4) * L.own_n * b);            // eta, grad, beta0, grad0 of the owned run
  L.total = off;
  return L;
}

template <typename AT>
__global__ void __launch_bounds__(kThreads, 1) small_kernel(const SmallArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int S = A.S, p = A.p, C = A.C;
  const uint32_t rank = S > 1 ? cluster_rank() : 0u;
  const int chain = int(blockIdx.x) / S;
  const Layout Lo = layout(A.n, p, C, S, sizeof(AT));
  AT* xs = reinterpret_cast<AT*>(smem + Lo.x);
  AT* beta = reinterpret_cast<AT*>(smem + Lo.beta);
  AT* recv = reinterpret_cast<AT*>(smem + Lo.recv);
  AT* z = reinterpret_cast<AT*>(smem + Lo.z);
  AT* rm = reinterpret_cast<AT*>(smem + Lo.rowv);
  AT* re = rm + Lo.rows;
  int* ys = reinterpret_cast<int*>(re + Lo.rows);
  AT* eta = reinterpret_cast<AT*>(smem + Lo.own);
  AT* grad = eta + Lo.own_n;
  AT* beta0 = grad + Lo.own_n;
  AT* grad0 = beta0 + Lo.own_n;
  double* scal = reinterpret_cast<double*>(smem + Lo.scal);         // rank 0: [S][4] sums of the CTAs
  double* decision = scal + 16 * 4;                                  // accept flag of the iteration
  double* wsum = decision + 8;                                       // [warps][4]
  const int pitch = Lo.pitch, own_n = Lo.own_n, E = C * p;
  const int e0 = int(rank) * own_n, ne = max(0, min(own_n, E - e0));   // owned coefficients
  const int64_t row0 = int64_t(rank) * Lo.rows;
  const int rows = int(max(int64_t(0), min(int64_t(Lo.rows), A.n - row0)));
  const bool zl = A.zlogit != 0;
  auto sync = [&]() {
    if (S > 1) cluster_sync_all();
    else __syncthreads();
  };

  // Element e (class e / p, feature e % p) of a buffer of rows of `ld`, one chain per `stride`.
  auto at = [&](int e, int64_t ld, int64_t stride) {
    const int k = e / p;
    return size_t(chain) * stride + size_t(k) * ld + (e - k * p);
  };
  const AT* gb = static_cast<const AT*>(A.beta);
  for (int e = tid; e < E; e += kThreads) beta[e] = gb[at(e, A.ld, A.stride)];
  for (int e = tid; e < ne; e += kThreads) {
    const size_t i = at(e0 + e, A.ld, A.stride);
    if (A.mode == kSmallLeap) eta[e] = static_cast<const AT*>(A.eta)[i];
    if (A.have_grad) grad[e] = static_cast<const AT*>(A.grad)[i];
  }
  {
    // Eight loads in flight per thread: filling 125 KB took 24 us with one.
    const AT* X = static_cast<const AT*>(A.X) + size_t(row0) * A.x_ld;
    const int total = rows * p;
    for (int b = tid; b < total; b += 8 * kThreads) {
      AT v[8];
      int d[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int e = b + i * kThreads, r = e / p, j = e - r * p;
        d[i] = r * pitch + j;
        v[i] = e < total ? X[size_t(r) * A.x_ld + j] : AT(0);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (b + i * kThreads < total) xs[d[i]] = v[i];
    }
  }
  for (int r = tid; r < rows; r += kThreads) ys[r] = A.y[row0 + r];
  sync();               // every CTA runs before any pushes into it

  // Lanes sharing one task (log2), so that enough threads have work.  FP64 issues 2
  // lanes a clock and SM, so six warps keep its units busy and every further butterfly
  // step costs what it adds; FP32 is bound by latency: all threads.
  auto lanes_for = [](int tasks) {
    constexpr int kWant = sizeof(AT) == 8 ? 192 : kThreads;
    int g = 0;
    while (g < 5 && (tasks << (g + 1)) <= kWant) ++g;
    return g;
  };
  // A thread's tasks t = (block, item), item fastest, of the two contractions: its first
  // one, found once (integer divisions take longer than the arithmetic of a small
  // step), and the tasks handled per pass.
  struct Walk {
    int g, ng, blk, item;
  };
  auto walk = [&](int tasks, int items) {
    Walk w;
    w.g = lanes_for(tasks);
    w.ng = kThreads >> w.g;
    const int t = tid >> w.g;
    w.blk = t / max(items, 1);
    w.item = t - w.blk * items;
    return w;
  };
  const AT s2 = AT(A.prior_scale * A.prior_scale);
  const int cblk = (C + kCB - 1) / kCB;
  const Walk wz = walk(cblk * rows, rows), wg = walk(cblk * p, p);
  int rw = 32;                     // threads that take a row each, a power of two
  while (rw < rows && rw < kThreads) rw *= 2;
  const int rsh = 31 - __clz(rw);
  const float inv_own = 1.f / float(own_n);
  auto owner_of = [&](int e) {     // e / own_n (e < 2^20: the estimate is off by one at most)
    int o = int(float(e) * inv_own);
    if (o * own_n > e) --o;
    if ((o + 1) * own_n <= e) ++o;
    return o;
  };
  double ll = 0.0;      // row log-likelihoods of this thread's rows (of the last gradient that wanted them)

  // Gradient of the likelihood at `beta`: partials of every owner's run land in its recv;
  // want_ll: the row log-likelihoods too (a logarithm per row, needed at a trajectory's end).
  auto partial_gradient = [&](bool want_ll) {
    {
      const int tasks = cblk * rows, G = 1 << wz.g, gl = tid & (G - 1);
      int cb = wz.blk, r = wz.item, t = tid >> wz.g;
      for (int t0 = 0; t0 < tasks; t0 += wz.ng) {
        const bool on = t < tasks;
        const int c0 = cb * kCB;
        AT a[kCB];
#pragma unroll
        for (int i = 0; i < kCB; ++i) a[i] = AT(0);
        const int nc = min(kCB, C - c0);
        if (on) dots_n(nc, a, xs + r * pitch, 1, beta + c0 * p, p, gl, p, G);
        for (int o = 1; o < G; o <<= 1)
#pragma unroll
          for (int i = 0; i < kCB; ++i)
            if (i < C) a[i] += __shfl_xor_sync(0xffffffffu, a[i], o);
        if (on && gl == 0)
#pragma unroll
          for (int i = 0; i < kCB; ++i)
            if (i < nc) z[(c0 + i) * rows + r] = a[i];
        t += wz.ng;
        for (r += wz.ng; r >= rows && cb < cblk; r -= rows) ++cb;
      }
    }
    __syncthreads();
    if constexpr (sizeof(AT) == 4) {
      // One thread per row.
      ll = 0.0;
      for (int r = tid; r < rows; r += kThreads) {
        const int yi = ys[r];
        float m = zl ? 0.f : -INFINITY;
        for (int k = 0; k < C; ++k) m = fmaxf(m, z[k * rows + r]);
        const float zy = yi < C ? z[yi * rows + r] : 0.f;      // yi == C: class K, logit 0
        float s = zl ? expf(-m) : 0.f;
        for (int k = 0; k < C; ++k) {
          const float e = expf(z[k * rows + r] - m);
          z[k * rows + r] = e;
          s += e;
        }
        const float inv = 1.f / s;
        for (int k = 0; k < C; ++k) z[k * rows + r] = (k == yi ? 1.f : 0.f) - z[k * rows + r] * inv;
        if (want_ll) ll += double(zy - m - logf(s));
      }
    } else {
      // The row's maximum, one exponential per (row, class), the row's sum, one residual
      // per (row, class): an FP64 exponential is a chain of some 35 operations.
      for (int r = tid; r < rows; r += kThreads) {
        AT m = zl ? AT(0) : AT(-INFINITY);
        for (int k = 0; k < C; ++k) m = max(m, z[k * rows + r]);
        rm[r] = m;
      }
      __syncthreads();
      ll = 0.0;
      if (want_ll)
        for (int r = tid; r < rows; r += kThreads)
          ll += double((ys[r] < C ? z[ys[r] * rows + r] : AT(0)) - rm[r]);   // label C: class K, logit 0
      if (want_ll) __syncthreads();
      for (int r = tid & (rw - 1); r < rows; r += rw)
        for (int k = tid >> rsh; k < C + (zl ? 1 : 0); k += kThreads >> rsh) {
          AT* d = k < C ? z + k * rows + r : re + r;
          *d = ex<AT>((k < C ? *d : AT(0)) - rm[r]);
        }
      __syncthreads();
      for (int r = tid; r < rows; r += kThreads) {
        AT s = zl ? re[r] : AT(0);
        for (int k = 0; k < C; ++k) s += z[k * rows + r];
        rm[r] = AT(1) / s;
        if (want_ll) ll -= double(lg<AT>(s));
      }
      __syncthreads();
      for (int r = tid & (rw - 1); r < rows; r += rw)
        for (int k = tid >> rsh; k < C; k += kThreads >> rsh)
          z[k * rows + r] = (k == ys[r] ? AT(1) : AT(0)) - z[k * rows + r] * rm[r];
    }
    __syncthreads();
    {
      const int tasks = cblk * p, G = 1 << wg.g, gl = tid & (G - 1);
      int cb = wg.blk, j = wg.item, t = tid >> wg.g;
      for (int t0 = 0; t0 < tasks; t0 += wg.ng) {
        const bool on = t < tasks;
        const int c0 = cb * kCB;
        AT a[kCB];
#pragma unroll
        for (int i = 0; i < kCB; ++i) a[i] = AT(0);
        const int nc = min(kCB, C - c0);
        if (on) dots_n(nc, a, xs + j, pitch, z + c0 * rows, rows, gl, rows, G);
        for (int o = 1; o < G; o <<= 1)
#pragma unroll
          for (int i = 0; i < kCB; ++i)
            if (i < C) a[i] += __shfl_xor_sync(0xffffffffu, a[i], o);
        if (on && gl == 0)
#pragma unroll
          for (int i = 0; i < kCB; ++i)
            if (i < nc) {
              const int e = (c0 + i) * p + j, o = owner_of(e);
              AT* d = recv + int(rank) * own_n + (e - o * own_n);
              if (S == 1) *d = a[i];
              else st_peer(map_peer(smem_u32(d), uint32_t(o)), a[i]);
            }
        t += wg.ng;
        for (j += wg.ng; j >= p && cb < cblk; j -= p) ++cb;
      }
    }
    sync();
  };
  // Gradient of the log posterior at owned coefficient e (prior included).
  auto full_gradient = [&](int e) {
    // Pairs, then pairs of pairs: the chain of additions stays short.
    AT v[16];
#pragma unroll
    for (int s = 0; s < 16; ++s) v[s] = s < S ? recv[s * own_n + e] : AT(0);
#pragma unroll
    for (int h = 1; h < 16; h *= 2)
      if (h < S)
#pragma unroll
        for (int s = 0; s < 16; s += 2 * h) v[s] += v[s + h];
    return v[0] + prior_deriv(beta[e0 + e], A.prior_kind, s2);
  };
  auto set_beta = [&](int e, AT v) {       // owned coefficient e, in every CTA
    AT* d = beta + e0 + e;
    if (S == 1) {
      *d = v;
    } else {
      const uint32_t a = smem_u32(d);
      for (int r = 0; r < S; ++r) st_peer(map_peer(a, uint32_t(r)), v);
    }
  };
  // Sums of four doubles over the cluster, in a fixed order; valid in thread 0 of rank 0.
  auto cluster_sums = [&](double (&v)[4]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane == 0)
#pragma unroll
      for (int k = 0; k < 4; ++k) wsum[warp * 4 + k] = v[k];
    __syncthreads();
    if (tid < 4) {
      double t = 0.0;
      for (int w = 0; w < kThreads / 32; ++w) t += wsum[w * 4 + tid];
      double* d = scal + int(rank) * 4 + tid;
      if (S == 1) *d = t;
      else st_peer(map_peer(smem_u32(d), 0u), t);
    }
    sync();
    if (rank == 0 && tid == 0)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        double t = 0.0;
        for (int s = 0; s < S; ++s) t += scal[s * 4 + k];
        v[k] = t;
      }
  };
  const AT half = AT(0.5 * A.eps), full = AT(A.eps);

  if (A.mode != kSmallSample) {
    double sums[4] = {0.0, 0.0, 0.0, 0.0};
    if (!A.have_grad || A.mode == kSmallGrad || A.L == 0) {
      partial_gradient(true);
      for (int e = tid; e < ne; e += kThreads) {
        grad[e] = full_gradient(e);
        sums[1] += prior_term(beta[e0 + e], A.prior_kind, A.prior_scale);
      }
      sums[0] = ll;
    }
    if (A.mode == kSmallLeap && A.L > 0) {
      sync();              // every owner has read its coefficients' partials and states
      for (int e = tid; e < ne; e += kThreads) {
        const AT v = eta[e] + half * grad[e];
        eta[e] = v;
        set_beta(e, beta[e0 + e] + full * v);
      }
      sync();
      for (int l = 1; l <= A.L; ++l) {
        partial_gradient(l == A.L);
        sums[0] = ll;
        sums[1] = 0.0;
        for (int e = tid; e < ne; e += kThreads) {
          const AT g = full_gradient(e), b = beta[e0 + e];
          const AT v = eta[e] + (l < A.L ? full : half) * g;
          eta[e] = v;
          grad[e] = g;
          if (l < A.L) set_beta(e, b + full * v);
          else sums[1] += prior_term(b, A.prior_kind, A.prior_scale);
        }
        sync();
      }
    }
    for (int e = tid; e < ne; e += kThreads) {
      const size_t i = at(e0 + e, A.ld, A.stride);
      if (A.mode == kSmallLeap) {
        static_cast<AT*>(A.beta_out)[i] = beta[e0 + e];
        static_cast<AT*>(A.eta)[i] = eta[e];
      }
      if (A.grad) static_cast<AT*>(A.grad)[i] = grad[e];
    }
    // The masked row K of user buffers is zero.
    if (A.ku > C)
      for (int j = int(rank) * kThreads + tid; j < p; j += S * kThreads) {
        const size_t i = size_t(chain) * A.stride + size_t(C) * A.ld + j;
        if (A.mode == kSmallLeap) {
          static_cast<AT*>(A.beta_out)[i] = AT(0);
          static_cast<AT*>(A.eta)[i] = AT(0);
        }
        if (A.grad) static_cast<AT*>(A.grad)[i] = AT(0);
      }
    if (A.logk) {
      cluster_sums(sums);
      if (rank == 0 && tid == 0) A.logk[chain] = sums[0] + sums[1];
    }
    if (S > 1) cluster_sync_all();   // no CTA leaves while a peer may still push into it
    return;
  }

  // ------------------------------------------------------------------ sampling
  const uint64_t it0 = uint64_t(*A.iter), seed = *A.seed;
  double logk = A.logk[chain];       // used by thread 0 of rank 0
  hmc_chain_stats st{};
  if (rank == 0 && tid == 0) st = static_cast<hmc_chain_stats*>(A.stats)[chain];
  for (int t = 0; t < A.iters; ++t) {
    double sums[4] = {0.0, 0.0, 0.0, 0.0};   // log-likelihood, prior, kinetic energy at the end and at the start
    for (int q = tid; q < (ne + 3) / 4; q += kThreads) {
      double mz[4];
      momentum_block(seed, it0 + uint64_t(t), uint64_t(chain), uint64_t((e0 >> 2) + q), mz);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = 4 * q + i;
        if (e < ne) {
          const AT m = AT(mz[i]), b = beta[e0 + e], g = grad[e];
          sums[3] += double(m) * double(m);
          beta0[e] = b;
          grad0[e] = g;
          const AT v = m + half * g;
          eta[e] = v;
          set_beta(e, b + full * v);
        }
      }
    }
    sync();
    for (int l = 1; l <= A.L; ++l) {
      partial_gradient(l == A.L);
      for (int e = tid; e < ne; e += kThreads) {
        const AT g = full_gradient(e), b = beta[e0 + e];
        const AT v = eta[e] + (l < A.L ? full : half) * g;
        eta[e] = v;
        grad[e] = g;
        if (l < A.L) {
          set_beta(e, b + full * v);
        } else {
          sums[1] += prior_term(b, A.prior_kind, A.prior_scale);
          sums[2] += double(v) * double(v);
        }
      }
      if (l < A.L) sync();
    }
    sums[0] = ll;
    cluster_sums(sums);
    if (rank == 0 && tid == 0) {
      const double lk1 = sums[0] + sums[1], h0 = -logk + 0.5 * sums[3], h1 = -lk1 + 0.5 * sums[2];
      const double T = A.temps ? A.temps[A.local0 + t] : 1.0;
      const bool finite = isfinite(h1);
      const double u = accept_uniform(seed, it0 + uint64_t(t), uint64_t(chain));
      const bool acc = finite && (log(u) < (h0 - h1) / T);
      st.iterations += 1;
      st.accepted += acc ? 1 : 0;
      st.diverged += finite ? 0 : 1;
      if (finite) st.sum_abs_dH += fabs(h1 - h0);
      if (acc) logk = lk1;
      st.logpost = logk;
      const double f = acc ? 1.0 : 0.0;
      if (S == 1) *decision = f;
      else
        for (int r = 0; r < S; ++r) st_peer(map_peer(smem_u32(decision), uint32_t(r)), f);
    }
    sync();
    const bool acc = *decision != 0.0;
    const int64_t li = A.local0 + t;
    AT* out = nullptr;
    if (A.samples && (li + 1) % A.thin == 0)
      out = static_cast<AT*>(A.samples) + size_t((li + 1) / A.thin - 1) * A.sample_stride + size_t(chain) * A.ku * p;
    for (int e = tid; e < ne; e += kThreads) {
      AT b = beta[e0 + e];
      if (!acc) {
        b = beta0[e];
        grad[e] = grad0[e];
        set_beta(e, b);
      }
      if (out) out[e0 + e] = b;        // rows of p: element e of the free rows in order
    }
    if (out && A.ku > C)
      for (int j = int(rank) * kThreads + tid; j < p; j += S * kThreads) out[size_t(C) * p + j] = AT(0);
    sync();
  }
  for (int e = tid; e < ne; e += kThreads) {
    const size_t i = at(e0 + e, A.ld, A.stride);
    static_cast<AT*>(A.beta_out)[i] = beta[e0 + e];
    static_cast<AT*>(A.grad)[i] = grad[e];
  }
  if (rank == 0 && tid == 0) {
    A.logk[chain] = logk;
    static_cast<hmc_chain_stats*>(A.stats)[chain] = st;
    // The last chain to finish advances the iteration counter (all have read it).
    __threadfence();
    if (atomicAdd(A.ticket, 1u) == unsigned(gridDim.x / S) - 1u) {
      *A.ticket = 0u;
      *A.iter = int64_t(it0) + A.iters;
    }
  }
  if (S > 1) cluster_sync_all();
}

// us of one gradient on a cluster of S CTAs: the two contractions (shared-memory bound
// in FP32, about 48 multiplies per ns and CTA; FP64 units 3.8), the exponentials (FP64
// about 40 operations each) and the barriers.
double step_us(bool f64, int64_t n, int64_t p, int64_t C, int S) {
  const double rows = double((n + S - 1) / S);
  const double fma = 2.0 * rows * double(p) * double(C), exps = rows * double(C + 1);
  return fma / (f64 ? 3800.0 : 48000.0) + exps * (f64 ? 0.0105 : 0.0005) + (S > 1 ? 1.5 : 0.5);
}

}  // namespace small

bool small_plan(int xt, int64_t n, int64_t p, int64_t C, int chains, int nsm, int smem_max, SmallPlan* out) {
  const bool f64 = xt == HMC_F64;
  if ((xt != HMC_F64 && xt != HMC_F32) || n < 1 || n > 16 * 1024 || C * p > (int64_t(1) << 20)) return false;
  SmallPlan best{};
  for (int S : {1, 2, 4, 8, 16}) {
    if (S > 1 && n < 2 * S) break;
    const small::Layout L = small::layout(n, int(p), int(C), S, f64 ? 8 : 4);
    if (L.total > size_t(smem_max)) continue;
    const int waves = (chains * S + nsm - 1) / nsm;
    const double us = small::step_us(f64, n, p, C, S) * waves;
    if (!best.S || us < best.us) best = SmallPlan{S, L.total, us};
  }
  if (!best.S) return false;
  *out = best;
  return true;
}

static const void* small_fn(int xt) {
  return xt == HMC_F64 ? reinterpret_cast<const void*>(small::small_kernel<double>)
                       : reinterpret_cast<const void*>(small::small_kernel<float>);
}

static void small_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int clusters, const SmallPlan& P,
                         cudaStream_t s) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3(clusters * P.S, 1, 1);
  cfg.blockDim = dim3(small::kThreads, 1, 1);
  cfg.dynamicSmemBytes = P.smem;
  cfg.stream = s;
  cfg.attrs = attr;
  if (P.S > 1) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = P.S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.numAttrs = 1;
  }
}

cudaError_t small_prepare(int xt, const SmallPlan& P, bool* fits) {
  *fits = false;
  int dev = 0, smem_max = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(small_fn(xt), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(small_fn(xt), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  int clusters = 1;
  if (P.S > 1) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    small_config(cfg, attr, 1, P, nullptr);
    if (cudaOccupancyMaxActiveClusters(&clusters, small_fn(xt), &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
  }
  *fits = clusters > 0;
  return cudaSuccess;
}

cudaError_t small_launch(int xt, const SmallPlan& P, const SmallArgs& a, int chains, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  small_config(cfg, attr, chains, P, s);
  if (xt == HMC_F64) return cudaLaunchKernelEx(&cfg, small::small_kernel<double>, a);
  return cudaLaunchKernelEx(&cfg, small::small_kernel<float>, a);
}

}  // namespace hmc
