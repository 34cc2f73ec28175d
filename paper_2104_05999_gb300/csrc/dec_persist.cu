// dec_persist.cu - the mixed-precision PCG of one instance as a single
// persistent kernel (cooperative launch: every block is resident).
//
// The solve is the one of the mixed mode in dec_solver.cu: CG with FP32
// vectors and L, a BF16 FSAI factor (or FP32 Jacobi), and FP64 defect
// correction by reliable updates (x64 += x32, r = b - L x64 in FP64 each time
// the FP32 residual has dropped by 1e-2; convergence decided in FP64).  The
// phases of an iteration are separated by a grid barrier instead of kernel
// boundaries, and every reduction ends with all blocks summing the block
// partials in the same order, so each block holds the same alpha, beta and
// residuals and takes the same branch without a host round trip.
//
// The barrier spins on a generation counter with a bounded number of polls;
// when the bound is hit the kernel records DEC_ERR_TIMEOUT and every block
// leaves at its next barrier.  Words 2 and 3 of the barrier (zero in normal
// use) let a test shorten the bound and withhold a block, so that this
// failure path runs without any endless wait.
#include "dec_kern.cuh"

#include <algorithm>
#include <cooperative_groups.h>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <utility>

namespace dec {

constexpr long kSpinLimit = 1L << 24;   // polls of 32-256 ns: a few seconds
// One block of 1024 threads per SM: fewer blocks make the grid barrier and
// the all-blocks partial sums cheaper (they cost per block, not per thread).
constexpr int kPBlock = 1024;

struct PersistArgs {
  int64_t n;
  SellArg<float> A32;
  SellArg<double> A64;
  SellArg<__nv_bfloat16> Glo, Gup;
  const float* dinv;          // Jacobi, or nullptr for FSAI
  const double* b;
  double *x64, *r64;
  float *x, *r, *z, *p, *q, *t;
  float *r2, *p2;             // second buffers of r and p
  double* partial;            // [4][gridDim.x]
  unsigned* bar;              // [0] arrivals, [1] generation
  int* status;                // [0] error, [1] iterations, [2] outcome
  double* result;             // [0] final rr (FP64), [1] |b|^2
  double rtol2, seg2;
  int max_iter;
};

// Grid barrier with a bounded spin.  Returns false once any block has
// timed out (then every block leaves).
__device__ __forceinline__ bool grid_sync(unsigned* bar, int* err) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u);
    if (arrived == gridDim.x - 1) {
      bar[0] = 0u;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      // bar[2] != 0 replaces the poll limit (the context's barrier test)
      const unsigned lim = *(volatile unsigned*)(bar + 2);
      const long limit = lim ? (long)lim : kSpinLimit;
      long polls = 0;
      unsigned ns = 32;
      while (*gen == g) {
        if (++polls > limit || *(volatile int*)err) {
          atomicExch(err, 1);
          break;
        }
        __nanosleep(ns);
        if (ns < 256) ns <<= 1;
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *(volatile int*)err == 0;
}

// Sum of NV (<= 2) per-thread values over the grid, identical in every
// block.  Consecutive calls alternate between two partial buffers: a block
// may write the partials of one sum while a slower block still reads those
// of the previous one, but never those of the one before (a barrier lies in
// between).  FP32 contributions (T = float) are added in FP32 inside each
// warp; everything above the warp level is FP64 and done by warp 0 alone
// (GB300's FP64 pipe is narrow, so FP64 work by every warp would dominate).
template <int NV, typename T>
__device__ __forceinline__ bool grid_sum(const T (&v)[NV], double (&tot)[NV],
                                         double* partial, int& parity, unsigned* bar,
                                         int* err) {
  __shared__ double sh[kPBlock];
  __shared__ double bc[2];
  double* part = partial + (size_t)parity * 2 * gridDim.x;
  parity ^= 1;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    double s;
    if constexpr (sizeof(T) == 4) s = block_sum_f<kPBlock>(v[k], sh);
    else s = block_sum<kPBlock>(v[k], sh);
    if (threadIdx.x == 0) part[k * gridDim.x + blockIdx.x] = s;
  }
  if (!grid_sync(bar, err)) return false;
  if (threadIdx.x < 32) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const double t = warp0_sum_array(part + k * gridDim.x, (int)gridDim.x);
      if (threadIdx.x == 0) bc[k] = t;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) tot[k] = bc[k];
  __syncthreads();
  return true;
}

// Row sum over the lane's row of slice s with the gathered operand formed on
// the fly: sum_j a_j * (X[c_j] + coef * Y[c_j]).  Used to fuse the vector
// update that produced the operand into the product that consumes it (the
// owner of row c computes the same fmaf for its own entry, so both agree).
template <typename MT>
__device__ __forceinline__ float sell_row2(const SellArg<MT>& A, int64_t s, int lane,
                                           const float* X, const float* Y, float coef) {
  constexpr int U = 8;
  const int32_t base = __ldg(A.sptr + s);
  const int32_t w = (__ldg(A.sptr + s + 1) - base) >> 5;
  const int32_t* __restrict__ cp = A.col + base + lane;
  const MT* __restrict__ vp = A.val + base + lane;
  float acc = 0.0f;
  for (int32_t j = 0; j < w; j += U) {
    int32_t c[U];
    MT av[U];
    float xv[U], yv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool ok = j + u < w;
      c[u] = ok ? __ldg(cp + 32 * (j + u)) : 0;
      av[u] = ok ? vp[32 * (j + u)] : MT(0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      xv[u] = j + u < w ? X[c[u]] : 0.0f;
      yv[u] = j + u < w ? Y[c[u]] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (j + u < w) acc = fma_(av[u], fmaf(coef, yv[u], xv[u]), acc);
  }
  return acc;
}

// One CG iteration is three phases separated by the three grid reductions
// it needs (p.q, r.r, r.z):
//   A: p_k = z + beta p_{k-1} (own rows) and q = L p_k, gathering z and
//      p_{k-1} so that p_k need not be complete first;
//   B: r_{k+1} = r_k - alpha q, x += alpha p_k (own rows) and t = G r_{k+1},
//      gathering r_k and q;
//   C: z = G^T t and r.z.
// p and r alternate between two buffers (a phase gathers the old vector while
// owners write the new one).  With Jacobi, B computes z = r / diag directly
// and C disappears.
template <bool JACOBI>
__global__ void __launch_bounds__(kPBlock, 1)
pcg_mixed_persistent(PersistArgs a) {
  // barrier test: bar[3] != 0 withholds the last block, so the others'
  // first barrier wait runs out (DEC_ERR_TIMEOUT)
  if (*(volatile unsigned*)(a.bar + 3) && blockIdx.x == gridDim.x - 1) return;
  const int64_t n = a.n;
  const int64_t gtid = blockIdx.x * (int64_t)kPBlock + threadIdx.x;
  const int64_t gstride = (int64_t)gridDim.x * kPBlock;
  const int lane = threadIdx.x & 31;
  const int64_t gwarp = gtid >> 5, nwarps = gstride >> 5;
  int* err = a.status;
  __shared__ float s_scal;
  __shared__ int s_flag;
  auto finish = [&](int outcome, int iters, double rr, double bb) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      a.status[1] = iters;
      a.status[2] = outcome;
      a.result[0] = rr;
      a.result[1] = bb;
    }
  };
  float* P[2] = {a.p, a.p2};
  float* R[2] = {a.r, a.r2};
  int cur = 0;
  // one slice per warp at a time; the gathered operand is X[c] (+ coef *
  // Y[c] when Y is given).  (Interleaving two slices per warp needed more
  // than the 64 registers a 1024-thread block allows and ran slower.)
  auto slices = [&](const auto& A, auto&& body, const float* X, const float* Y, float coef) {
    for (int64_t s = gwarp; s < A.nslices; s += nwarps) {
      const float acc = Y ? sell_row2(A, s, lane, X, Y, coef) : sell_row(A, s, lane, X);
      const int32_t r0 = __ldg(A.perm + 32 * s + lane);
      if (r0 >= 0) body(r0, acc);
    }
  };

  // ---- start: x64 = 0, r64 = b, r = (float) b, x = p = 0
  int parity = 0;
  double v1[1], t1[1];
  {
    double bb = 0.0;
    for (int64_t i = gtid; i < n; i += gstride) {
      const double bi = a.b[i];
      a.x64[i] = 0.0;
      a.r64[i] = bi;
      a.r[i] = (float)bi;
      a.x[i] = 0.0f;
      a.p[i] = 0.0f;
      a.p2[i] = 0.0f;
      bb += bi * bi;
    }
    v1[0] = bb;
  }
  if (!grid_sum<1>(v1, t1, a.partial, parity, a.bar, err)) return;
  const double bnorm2 = t1[0];
  if (bnorm2 == 0.0) { finish(0, 0, 0.0, 0.0); return; }
  double rr64 = bnorm2, best = bnorm2, rz = 0.0;
  double tol2 = a.seg2 * rr64;
  int iters = 0, stall = 0, restart = 1;
  float beta = 0.0f;

  for (;;) {
    // ---- segment start: z = M r (from R[cur]), r.z, beta
    {
      float v[1] = {0.0f};
      double t[1];
      const float* rc = R[cur];
      if (JACOBI) {
        float acc = 0.0f;
        for (int64_t i = gtid; i < n; i += gstride) {
          const float zi = a.dinv[i] * rc[i];
          a.z[i] = zi;
          acc = fmaf(rc[i], zi, acc);
        }
        v[0] = acc;
      } else {
        slices(a.Glo, [&](int32_t row, float acc) { a.t[row] = acc; }, rc,
              (const float*)nullptr, 0.0f);
        if (!grid_sync(a.bar, err)) return;
        float acc2 = 0.0f;
        slices(a.Gup, [&](int32_t row, float acc) {
          a.z[row] = acc;
          acc2 = fmaf(rc[row], acc, acc2);
        }, a.t, (const float*)nullptr, 0.0f);
        v[0] = acc2;
      }
      if (!grid_sum<1>(v, t, a.partial, parity, a.bar, err)) return;
      if (threadIdx.x == 0) s_scal = (restart || rz == 0.0) ? 0.0f : (float)(t[0] / rz);
      __syncthreads();
      beta = s_scal;
      rz = t[0];
    }
    // ---- FP32 iterations until the residual has dropped by seg2
    int breakdown = 0;
    for (;;) {
      const int nxt = cur ^ 1;
      // A: p_k = z + beta p_{k-1}, q = L p_k, p_k . q
      {
        const float* pold = P[cur];
        float* pnew = P[nxt];
        float acc2 = 0.0f;
        slices(a.A32, [&](int32_t row, float qi) {
          const float pi = fmaf(beta, pold[row], a.z[row]);
          pnew[row] = pi;
          a.q[row] = qi;
          acc2 = fmaf(pi, qi, acc2);
        }, a.z, pold, beta);
        float vq[1] = {acc2};
        double tq[1];
        if (!grid_sum<1>(vq, tq, a.partial, parity, a.bar, err)) return;
        if (threadIdx.x == 0) {
          const double pq = tq[0];
          s_flag = (!(pq > 0.0) || !isfinite(pq)) ? 1 : 0;
          s_scal = s_flag ? 0.0f : (float)(rz / pq);
        }
        __syncthreads();
      }
      if (s_flag) { breakdown = 1; cur = nxt; break; }   // p_k is in P[nxt]
      const float alpha = s_scal;
      // B: r_{k+1} = r_k - alpha q, x += alpha p_k, t = G r_{k+1}, r.r
      float rr = 0.0f, rzj = 0.0f;
      {
        const float* rold = R[cur];
        float* rnew = R[nxt];
        const float* pk = P[nxt];
        if (JACOBI) {
          for (int64_t i = gtid; i < n; i += gstride) {
            const float ri = fmaf(-alpha, a.q[i], rold[i]);
            rnew[i] = ri;
            a.x[i] = fmaf(alpha, pk[i], a.x[i]);
            rr = fmaf(ri, ri, rr);
            const float zi = a.dinv[i] * ri;
            a.z[i] = zi;
            rzj = fmaf(ri, zi, rzj);
          }
        } else {
          slices(a.Glo, [&](int32_t row, float ti) {
            const float ri = fmaf(-alpha, a.q[row], rold[row]);
            rnew[row] = ri;
            a.x[row] = fmaf(alpha, pk[row], a.x[row]);
            a.t[row] = ti;
            rr = fmaf(ri, ri, rr);
          }, rold, (const float*)a.q, -alpha);
        }
      }
      float v2[2] = {rr, rzj};
      double t2[2];
      if (!grid_sum<2>(v2, t2, a.partial, parity, a.bar, err)) return;
      cur = nxt;
      ++iters;
      if (t2[0] <= tol2 || iters >= a.max_iter || !isfinite(t2[0])) break;
      double rz_new;
      if (JACOBI) {
        rz_new = t2[1];
      } else {
        // C: z = G^T t, r.z
        float acc2 = 0.0f;
        const float* rcur = R[cur];
        slices(a.Gup, [&](int32_t row, float zi) {
          a.z[row] = zi;
          acc2 = fmaf(rcur[row], zi, acc2);
        }, a.t, (const float*)nullptr, 0.0f);
        float vz[1] = {acc2};
        double tz[1];
        if (!grid_sum<1>(vz, tz, a.partial, parity, a.bar, err)) return;
        rz_new = tz[0];
      }
      if (threadIdx.x == 0) s_scal = (float)(rz_new / rz);
      __syncthreads();
      beta = s_scal;
      rz = rz_new;
    }
    // ---- reliable update: x64 += x, x = 0; r64 = b - L x64; R[cur] = (float) r64
    for (int64_t i = gtid; i < n; i += gstride) {
      a.x64[i] += (double)a.x[i];
      a.x[i] = 0.0f;
    }
    if (!grid_sync(a.bar, err)) return;
    {
      double rr = 0.0;
      float* rc = R[cur];
      for (int64_t s = gwarp; s < a.A64.nslices; s += nwarps) {
        const int32_t row = __ldg(a.A64.perm + 32 * s + lane);
        const double acc = sell_row(a.A64, s, lane, a.x64);
        if (row >= 0) {
          const double ri = a.b[row] - acc;
          a.r64[row] = ri;
          rc[row] = (float)ri;
          rr = fma(ri, ri, rr);
        }
      }
      v1[0] = rr;
    }
    if (!grid_sum<1>(v1, t1, a.partial, parity, a.bar, err)) return;
    rr64 = t1[0];
    if (rr64 <= a.rtol2 * bnorm2) { finish(0, iters, rr64, bnorm2); return; }
    if (iters >= a.max_iter) { finish(1, iters, rr64, bnorm2); return; }
    if (rr64 < 0.5 * best) { best = rr64; stall = 0; }
    else if (++stall >= 4) { finish(2, iters, rr64, bnorm2); return; }
    restart = (breakdown || stall > 0) ? 1 : 0;
    tol2 = a.seg2 * rr64;
  }
}

// One mixed-precision solve of instance `inst` with the persistent kernel.
// Returns DEC_ERR_LIMIT when a cooperative launch is not possible (the
// caller then uses the kernel-per-phase path).
dec_status solve_mixed_persistent(dec_ctx* ctx, int inst, double rtol, int max_iter,
                                  int* iters_out, double* relres_out) {
  const int64_t n = ctx->n;
  const int vs = value_set(ctx, inst);
  cudaStream_t s = ctx->stream;
  const bool fsai = ctx->precond == DEC_PRECOND_FSAI;
  int dev_coop = 0;
  DEC_TRY(cudaDeviceGetAttribute(&dev_coop, cudaDevAttrCooperativeLaunch, ctx->device));
  if (!dev_coop) return DEC_ERR_LIMIT;
  auto kern = fsai ? pcg_mixed_persistent<false> : pcg_mixed_persistent<true>;
  int per_sm = 0;
  DEC_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPBlock, 0));
  if (per_sm < 1) return DEC_ERR_LIMIT;
  const int grid = ctx->num_sms;   // one block per SM (per_sm >= 1 checked)
  DEC_TRY(ctx->partial.ensure((size_t)kRedSlots * std::max(grid, ctx->reduce_grid)));
  DEC_TRY_STATUS(sell_copies(ctx, vs, 2));
  DEC_TRY(ctx->coop.ensure(16));
  unsigned* bar = reinterpret_cast<unsigned*>(ctx->coop.p);
  int* status = reinterpret_cast<int*>(ctx->coop.p + 2);
  double* result = reinterpret_cast<double*>(ctx->coop.p + 8);
  DEC_TRY(cudaMemsetAsync(ctx->coop.p, 0, 16 * sizeof(int64_t), s));
  DEC_TRY(write_barrier_test(ctx, bar));
  PersistArgs a{};
  a.n = n;
  a.A32 = sell_arg(ctx->sellL, ctx->sL32.p + (int64_t)vs * ctx->sellL.total);
  a.A64 = sell_arg(ctx->sellL, ctx->sL64.p + (int64_t)vs * ctx->sellL.total);
  a.Glo = sell_arg(ctx->sellLo, fsai ? ctx->sGlo16.p + (int64_t)vs * ctx->sellLo.total : nullptr);
  a.Gup = sell_arg(ctx->sellUp, fsai ? ctx->sGup16.p + (int64_t)vs * ctx->sellUp.total : nullptr);
  a.dinv = fsai ? nullptr : ctx->dinv32.p + (int64_t)vs * n;
  a.b = ctx->b.p + (int64_t)inst * n;
  a.x64 = ctx->u.p + (int64_t)inst * n;
  a.r64 = ctx->r64.p;
  a.x = ctx->x32.p; a.r = ctx->r32.p; a.z = ctx->z32.p; a.p = ctx->p32.p;
  a.q = ctx->q32.p; a.t = ctx->t32.p;
  DEC_TRY(ctx->r32b.ensure(n));
  DEC_TRY(ctx->p32b.ensure(n));
  a.r2 = ctx->r32b.p; a.p2 = ctx->p32b.p;
  a.partial = ctx->partial.p;
  a.bar = bar;
  a.status = status;
  a.result = result;
  a.rtol2 = rtol * rtol;
  a.seg2 = 1e-4;
  a.max_iter = max_iter;
  void* args[] = {&a};
  DEC_TRY(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kPBlock), args, 0, s));
  ctx->launches += 1;
  int hs[3];
  double hr[2];
  DEC_TRY(cudaMemcpyAsync(hs, status, sizeof(hs), cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaMemcpyAsync(hr, result, sizeof(hr), cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaStreamSynchronize(s));
  *iters_out = hs[1];
  *relres_out = hr[1] > 0.0 ? std::sqrt(hr[0] / hr[1]) : 0.0;
  if (hs[0]) return ctx->fail(DEC_ERR_TIMEOUT, "persistent solve: a grid barrier timed out");
  if (hs[2] == 1) return ctx->fail(DEC_NOT_CONVERGED, "max_iter reached");
  if (hs[2] == 2) return ctx->fail(DEC_NOT_CONVERGED, "residual replacement stalled");
  return DEC_OK;
}

// ------------------------------------------- FP64 PCG of small systems
// One cluster of 16 blocks runs the whole FP64 solve of up to
// kClusterRows nodes: the three phases per iteration of the kernel above,
// separated by cluster barriers, block sums exchanged through distributed
// shared memory.  Bound by latency: a phase is one round of gathers from L2,
// a sum in the block and a cluster barrier.  Whole solve to 1e-10 at 3,375
// nodes with FSAI, 47 iterations: 788 us (16.8 us an iteration, set-up and
// read-back included) against 1,415 us for five kernels per iteration in a
// graph; at 729 nodes 432 against 905 us.  Eight blocks that read the matrix
// from L2, two slices a warp, took 988 us.
constexpr int kCBlock = 512;
constexpr int kCBlocks = 16;

struct ClusterArgs {
  int64_t n;
  SellArg<double> A, Glo, Gup;
  const double* dinv;         // Jacobi, or nullptr for FSAI
  const double* b;
  double* x;                  // start (warm) and solution
  double *r[2], *p[2], *z, *q, *t;
  double rtol2;
  int max_iter, warm;
  int cap;                    // entries a block's shared memory holds
  int* status;                // [0] iterations, [1] 0 converged, 1 max_iter, 3 breakdown
  double* result;             // [0] |b - L x|^2, [1] |b|^2
};

// store v at block b's copy of the shared address `at`
__device__ __forceinline__ void store_cluster(uint32_t at, int b, double v) {
  asm volatile(
      "{\n\t.reg .b32 remote;\n\t"
      "mapa.shared::cluster.u32 remote, %0, %1;\n\t"
      "st.shared::cluster.f64 [remote], %2;\n\t}"
      :: "r"(at), "r"(b), "d"(v) : "memory");
}

template <bool JACOBI>
__global__ void __launch_bounds__(kCBlock, 1)
pcg_cluster_kernel(ClusterArgs a) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  // No block may store into another's shared memory before that one runs:
  // arrive here, wait after the matrix is staged, before the first sum.
  cg::cluster_group::arrival_token started = cluster.barrier_arrive();
  __shared__ double sh[2][kCBlock];
  __shared__ double slot[2][2][kCBlocks][32];   // [parity][value][block][lane]
  __shared__ double bc[3];                      // sums and a ratio for the whole block
  const int rank = (int)cluster.block_rank();
  const int64_t n = a.n;
  const int64_t gtid = (int64_t)rank * kCBlock + threadIdx.x;
  const int64_t gstride = (int64_t)kCBlocks * kCBlock;
  const int lane = threadIdx.x & 31;
  // consecutive slices on different SMs
  const int64_t gwarp = (int64_t)(threadIdx.x >> 5) * kCBlocks + rank;
  int parity = 0;
  // Sums of one or two values over the cluster, in a fixed order, into
  // bc[0..1] of every block; also the barrier between phases.  finish(s0, s1)
  // goes to bc[2].  One FP64 instruction of a warp holds the SM's pipe for 16
  // cycles, so one warp adds the block's values lane by lane, the 32 lane
  // sums of each block are exchanged, and only their total takes a butterfly.
  auto sum2 = [&](double v0, double v1, auto two_c, auto&& finish) {
    constexpr int NV = decltype(two_c)::value ? 2 : 1;
    sh[0][threadIdx.x] = v0;
    if constexpr (NV == 2) sh[1][threadIdx.x] = v1;
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        double t[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) t[c] = sh[k][32 * c + lane];
#pragma unroll
        for (int w = 4; w < kCBlock / 32; ++w) t[w & 3] += sh[k][32 * w + lane];
        const double own = (t[0] + t[1]) + (t[2] + t[3]);
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&slot[parity][k][rank][lane]);
#pragma unroll 4
        for (int b = 0; b < kCBlocks; ++b) store_cluster(mine, b, own);
      }
    }
    cluster.sync();
    if (threadIdx.x < 32) {
      double tot[2] = {0.0, 0.0};
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        double t[2] = {slot[parity][k][0][lane], slot[parity][k][1][lane]};
#pragma unroll
        for (int b = 2; b < kCBlocks; ++b) t[b & 1] += slot[parity][k][b][lane];
        tot[k] = t[0] + t[1];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], o);
      }
      if (lane == 0) {
        bc[0] = tot[0];
        bc[1] = tot[1];
        bc[2] = finish(tot[0], tot[1]);
      }
    }
    parity ^= 1;
    __syncthreads();
  };
  using One = std::false_type;
  using Two = std::true_type;
  auto nothing = [](double, double) { return 0.0; };
  // This warp's slice of each matrix.
  constexpr int kL = 0, kLo = 1, kUp = 2;
  extern __shared__ __align__(16) double cvals[];
  uint16_t* ccols = reinterpret_cast<uint16_t*>(cvals + a.cap);
  __shared__ int used;
  if (threadIdx.x == 0) used = 0;
  __syncthreads();
  int32_t off[3], wid[3], row_of[3];   // first slot + lane, width, this lane's row
  int32_t entries = 0;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const SellArg<double>& A = m == kL ? a.A : m == kLo ? a.Glo : a.Gup;
    const bool have = (m == kL || !JACOBI) && gwarp < A.nslices;
    off[m] = have ? __ldg(A.sptr + gwarp) + lane : 0;
    wid[m] = have ? (__ldg(A.sptr + gwarp + 1) - __ldg(A.sptr + gwarp)) >> 5 : 0;
    row_of[m] = have ? __ldg(A.perm + 32 * gwarp + lane) : -1;
    entries += 32 * wid[m];
  }
  int32_t at = 0;
  if (lane == 0) at = atomicAdd(&used, entries);
  at = __shfl_sync(0xffffffffu, at, 0) + lane;
  __syncthreads();
  // Entries in shared memory (16-bit columns) where a block's all fit: of the
  // three dependent trips to L2 per phase (column, operand, then the sum) the
  // operand's is left.
  const bool staged = used <= a.cap;
  if (staged) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const SellArg<double>& A = m == kL ? a.A : m == kLo ? a.Glo : a.Gup;
      for (int32_t j = 0; j < wid[m]; ++j) {
        cvals[at + 32 * j] = __ldg(A.val + off[m] + 32 * j);
        ccols[at + 32 * j] = (uint16_t)__ldg(A.col + off[m] + 32 * j);
      }
      off[m] = at;
      at += 32 * wid[m];
    }
    __syncwarp();
  }
  auto run = [&](auto staged_c) {
  constexpr bool STAGED = decltype(staged_c)::value;
  // For this warp's rows of matrix m: own(row) before the products,
  // body(row, product, own) after them; the operand is X[c] (TWO: X[c] +
  // coef Y[c]).  The loads of a round are issued before any is used.
  auto product = [&](auto two_c, auto m_c, const double* X, const double* Y, double coef,
                     auto&& own, auto&& body) {
    constexpr bool TWO = decltype(two_c)::value;
    constexpr int m = decltype(m_c)::value;
    constexpr int U = TWO ? 4 : 6;   // more spill registers at 512 threads: 24 ms, not 21.7
    const SellArg<double>& A = m == kL ? a.A : m == kLo ? a.Glo : a.Gup;
    const int32_t w = wid[m], row = row_of[m];
    double2 mine = make_double2(0.0, 0.0);
    if (row >= 0) mine = own(row);
    double acc = 0.0;
#pragma unroll 1
    for (int32_t j = 0; j < w; j += U) {
      double xv[U], yv[TWO ? U : 1];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (j + u < w) {
          const int32_t e = off[m] + 32 * (j + u);
          const int32_t c = STAGED ? (int32_t)ccols[e] : __ldg(A.col + e);
          xv[u] = X[c];
          if constexpr (TWO) yv[u] = Y[c];
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (j + u < w) {
          const int32_t e = off[m] + 32 * (j + u);
          const double v = STAGED ? cvals[e] : __ldg(A.val + e);
          if constexpr (TWO) acc = fma(v, fma(coef, yv[u], xv[u]), acc);
          else acc = fma(v, xv[u], acc);
        }
    }
    if (row >= 0) body(row, acc, mine);
  };
  using L0 = std::integral_constant<int, kL>;
  using LO = std::integral_constant<int, kLo>;
  using UP = std::integral_constant<int, kUp>;
  auto plain = [&](auto m_c, const double* X, auto&& own, auto&& body) {
    product(std::false_type{}, m_c, X, (const double*)nullptr, 0.0, own, body);
  };
  auto fused = [&](auto m_c, const double* X, const double* Y, double coef, auto&& own,
                   auto&& body) {
    product(std::true_type{}, m_c, X, Y, coef, own, body);
  };
  auto none = [](int32_t) { return make_double2(0.0, 0.0); };
  int cur = 0, pc = 0;
  // r = b - L x, r.r in bc[0]
  auto residual = [&]() {
    double rr = 0.0;
    double* r = a.r[cur];
    plain(L0{}, a.x, [&](int32_t row) { return make_double2(a.b[row], 0.0); },
          [&](int32_t row, double acc, double2 o) {
            const double ri = o.x - acc;
            r[row] = ri;
            rr = fma(ri, ri, rr);
          });
    sum2(rr, 0.0, One{}, nothing);
  };

  {
    double bb = 0.0;
    for (int64_t i = gtid; i < n; i += gstride) {
      const double bi = a.b[i];
      if (!a.warm) {
        a.x[i] = 0.0;
        a.r[0][i] = bi;
      }
      a.p[0][i] = 0.0;
      bb = fma(bi, bi, bb);
    }
    sum2(bb, 0.0, One{}, nothing);
  }
  const double bnorm2 = bc[0], tol2 = a.rtol2 * bnorm2;
  // Only b = 0, or a warm start that meets the tolerance, needs no iteration;
  // the host reports a right-hand side that is not finite.
  double rr = nan("");
  if (a.warm && bnorm2 > 0.0) {
    residual();
    rr = bc[0];
  }
  int iters = 0, outcome = 0;
  while (bnorm2 > 0.0 && !(rr <= tol2)) {
    // (re)start: z = M r, r.z, beta = 0
    double v = 0.0;
    const double* rc = a.r[cur];
    if (JACOBI) {
      for (int64_t i = gtid; i < n; i += gstride) {
        const double zi = a.dinv[i] * rc[i];
        a.z[i] = zi;
        v = fma(rc[i], zi, v);
      }
    } else {
      plain(LO{}, rc, none, [&](int32_t row, double acc, double2) { a.t[row] = acc; });
      cluster.sync();
      plain(UP{}, a.t, [&](int32_t row) { return make_double2(rc[row], 0.0); },
            [&](int32_t row, double acc, double2 o) {
              a.z[row] = acc;
              v = fma(o.x, acc, v);
            });
    }
    sum2(v, 0.0, One{}, nothing);
    double rz = bc[0], beta = 0.0;
    bool breakdown = false;
    for (;;) {
      // A: p = z + beta p, q = L p, p.q
      const double* po = a.p[pc];
      double* pn = a.p[pc ^ 1];
      double acc = 0.0;
      fused(L0{}, a.z, po, beta, [&](int32_t row) { return make_double2(po[row], a.z[row]); },
            [&](int32_t row, double qi, double2 o) {
              const double pi = fma(beta, o.x, o.y);
              pn[row] = pi;
              a.q[row] = qi;
              acc = fma(pi, qi, acc);
            });
      sum2(acc, 0.0, One{}, [&](double s, double) { return rz / s; });
      pc ^= 1;
      const double pq = bc[0], alpha = bc[2];
      if (!(pq > 0.0) || !isfinite(pq)) { breakdown = true; break; }
      // B: r' = r - alpha q, x += alpha p, r'.r', t = G r' (Jacobi: z, r'.z)
      const double* ro = a.r[cur];
      double* rn = a.r[cur ^ 1];
      double s0 = 0.0, s1 = 0.0;
      if constexpr (JACOBI) {
        for (int64_t i = gtid; i < n; i += gstride) {
          const double ri = fma(-alpha, a.q[i], ro[i]);
          rn[i] = ri;
          a.x[i] = fma(alpha, pn[i], a.x[i]);
          s0 = fma(ri, ri, s0);
          const double zi = a.dinv[i] * ri;
          a.z[i] = zi;
          s1 = fma(ri, zi, s1);
        }
      } else {
        fused(LO{}, ro, a.q, -alpha,
              [&](int32_t row) {
                return make_double2(fma(-alpha, a.q[row], ro[row]),
                                    fma(alpha, pn[row], a.x[row]));
              },
              [&](int32_t row, double ti, double2 o) {
                rn[row] = o.x;
                a.x[row] = o.y;
                a.t[row] = ti;
                s0 = fma(o.x, o.x, s0);
              });
      }
      sum2(s0, s1, std::bool_constant<JACOBI>{}, [&](double, double s) { return s / rz; });
      cur ^= 1;
      ++iters;
      rr = bc[0];
      if (rr <= tol2 || iters >= a.max_iter || !isfinite(rr)) break;
      if constexpr (JACOBI) {
        rz = bc[1];
      } else {
        // C: z = G^T t, r'.z
        double w = 0.0;
        plain(UP{}, a.t, [&](int32_t row) { return make_double2(rn[row], 0.0); },
              [&](int32_t row, double zi, double2 o) {
                a.z[row] = zi;
                w = fma(o.x, zi, w);
              });
        sum2(w, 0.0, One{}, [&](double s, double) { return s / rz; });
        rz = bc[0];
      }
      beta = bc[2];
    }
    // the true residual decides
    residual();
    rr = bc[0];
    if (breakdown) { outcome = 3; break; }
    if (rr <= tol2) break;
    if (iters >= a.max_iter) { outcome = 1; break; }
  }
  if (rank == 0 && threadIdx.x == 0) {
    a.status[0] = iters;
    a.status[1] = outcome;
    a.result[0] = bnorm2 > 0.0 ? rr : 0.0;
    a.result[1] = bnorm2;
  }
  };
  cluster.barrier_wait(std::move(started));   // every block of the cluster runs
  if (staged) run(std::true_type{});
  else run(std::false_type{});
  cluster.sync();     // no block leaves while another may write its slots
}

dec_status solve_fp64_cluster(dec_ctx* ctx, int inst, double rtol, int max_iter, bool warm,
                              int* iters_out, double* relres_out) {
  const int64_t n = ctx->n;
  const int vs = value_set(ctx, inst);
  cudaStream_t s = ctx->stream;
  const bool fsai = ctx->precond == DEC_PRECOND_FSAI;
  const int cap = 19 * 1024;  // 190 KB of values and 16-bit columns
  const int smem = cap * (int)(sizeof(double) + sizeof(uint16_t));
  auto kern = fsai ? pcg_cluster_kernel<false> : pcg_cluster_kernel<true>;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kCBlocks;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kCBlocks);
  cfg.blockDim = dim3(kCBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  // 16 blocks are above the portable cluster size: a device (or a part of
  // one) whose GPCs have fewer SMs to give cannot place such a cluster
  int& fits = ctx->cluster_fits[fsai];
  if (fits < 0) {
    int clusters = 0;
    const bool ok =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) ==
            cudaSuccess &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
            cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess;
    if (!ok) cudaGetLastError();
    fits = ok && clusters > 0 ? 1 : 0;
  }
  if (!fits) return DEC_ERR_LIMIT;
  DEC_TRY_STATUS(sell_copies(ctx, vs, 1));
  DEC_TRY(ctx->coop.ensure(16));
  DEC_TRY(ctx->p64b.ensure(n));
  DEC_TRY(ctx->r64b.ensure(n));
  ClusterArgs a{};
  a.n = n;
  a.A = sell_arg(ctx->sellL, ctx->sL64.p + (int64_t)vs * ctx->sellL.total);
  a.Glo = sell_arg(ctx->sellLo, fsai ? ctx->sGlo64.p + (int64_t)vs * ctx->sellLo.total : nullptr);
  a.Gup = sell_arg(ctx->sellUp, fsai ? ctx->sGup64.p + (int64_t)vs * ctx->sellUp.total : nullptr);
  a.dinv = fsai ? nullptr : ctx->dinv64.p + (int64_t)vs * n;
  a.b = ctx->b.p + (int64_t)inst * n;
  a.x = ctx->u.p + (int64_t)inst * n;
  a.r[0] = ctx->r64.p;
  a.r[1] = ctx->r64b.p;
  a.p[0] = ctx->p64.p;
  a.p[1] = ctx->p64b.p;
  a.z = ctx->z64.p;
  a.q = ctx->q64.p;
  a.t = ctx->t64.p;
  a.rtol2 = rtol * rtol;
  a.max_iter = max_iter;
  a.warm = warm ? 1 : 0;
  a.status = reinterpret_cast<int*>(ctx->coop.p + 2);
  a.result = reinterpret_cast<double*>(ctx->coop.p + 8);
  a.cap = cap;
  DEC_TRY(cudaLaunchKernelEx(&cfg, kern, a));
  DEC_TRY(cudaGetLastError());
  ctx->launches += 1;
  int64_t h[16];
  DEC_TRY(cudaMemcpyAsync(h, ctx->coop.p, sizeof(h), cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaStreamSynchronize(s));
  int hs[2];
  double hr[2];
  memcpy(hs, h + 2, sizeof(hs));
  memcpy(hr, h + 8, sizeof(hr));
  *iters_out = hs[0];
  *relres_out = hr[1] > 0.0 ? std::sqrt(hr[0] / hr[1]) : 0.0;
  if (hs[1] == 3 || !std::isfinite(hr[1]))
    return ctx->fail(DEC_ERR_BREAKDOWN, "CG breakdown: p.Lp <= 0 or not finite");
  if (hs[1] == 1) return ctx->fail(DEC_NOT_CONVERGED, "max_iter reached");
  return DEC_OK;
}

}  // namespace dec
