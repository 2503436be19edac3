// tg_cg_small.cu -- the FP64 Jacobi-CG solves of small grids as one launch each.
//
// On grids up to a few ten thousand voxels a CG iteration of the many-kernel form is latency:
// at 32^3 its three kernels carry 5 us of arithmetic and take 22 us, most of it launches,
// ramps and the last block's sum.  Here one cooperative kernel runs the whole solve.  Every
// thread owns one voxel and keeps the voxel's part of the CG vectors (increment, residual,
// direction, A p, inverse diagonal) in registers and its operator coefficients in shared
// memory from the first iteration to the last; only the preconditioned residual z goes through
// memory, for the neighbours' operator.  The operator is applied to z, and A p follows by the
// recurrence of the direction, p = z + beta p, A p = A z + beta A p: so an iteration has two
// grid-wide waits, each of which also carries sums (a block leaves its partial sums before the
// wait; after it one warp of every block adds all of them in block order, so every block takes
// the same decision with no further round trip), and none to publish the direction.
//
// One block per SM: the grid is dealt out in blocks of 32 ceil(n / (32 SMs)) threads, which
// spreads the FP64 work (75 operations of the elasticity operator per voxel, on a pipe of two
// lanes per clock and SM) evenly over the SMs; 512 threads of 128 registers fill an SM's
// register file and their 27 coefficients 108 KB of its shared memory, so grids up to 512
// voxels per SM (77824 on 152 SMs) take this form.
//
// Measured (three launches an iteration -> this form): a static solve at 16^3 590 -> 300 us, two
// FP64 steps at 32^3 2.70 -> 2.01 ms.  Near the size limit (69120 voxels) an iteration takes
// 20.4 us, 11.5 of them on the FP64 pipe; the rest is the two waits and the neighbours' z from L2.
//
// The waits are bounded in time (tg_wait.cuh; the context's limit, 20 s unless it is set): a
// block that gives up marks the solve CG_TIMEOUT and returns, the others give up in their turn
// or, if all arrived late, finish, and the solve stays marked either way.  Launched
// cooperatively, so all blocks are resident; the default limit is far above the microseconds of a
// wait for programs that keep other kernels, or other processes' time slices, on the same GPU.
#include <type_traits>

#include "tg_internal.cuh"

namespace tg {
namespace {

// Waits until all blocks of the launch have arrived for the round-th time (round = 1, 2, ...);
// everything any thread wrote before its block's arrival is visible after it (the barrier and
// the release of thread 0 order the block's writes before the arrival, its acquire and the
// second barrier order the others' before what follows).  False in every thread of the block if
// the wait ran out.
__device__ __forceinline__ bool grid_wait(unsigned int* words, unsigned int round,
                                          unsigned long long limit_ns) {
  __shared__ bool ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    wait_arrive(words);
    ok = wait_for_arrivals(words, round, gridDim.x, limit_ns);
  }
  __syncthreads();
  return ok;
}

// NV sums over the block's threads into partial[q * gridDim.x + block], one warp per value
template <int NV>
__device__ __forceinline__ void leave_partials(const double (&v)[NV], double* partial) {
  __shared__ double sh[NV][CGS_MAX_THREADS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int q = warp; q < NV; q += nw) {
    const double s = warp_sum_shared(sh[q], blockDim.x, lane);
    if (lane == 0) partial[(size_t)q * gridDim.x + blockIdx.x] = s;
  }
}

// the sum of one value's partials over all blocks, by one whole warp, valid in every lane
__device__ __forceinline__ double all_partials(const double* partial) {
  double s = strided_partials(partial, 1, gridDim.x, threadIdx.x & 31, 32);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// The operator's coefficients of one voxel, in shared memory: coefficient q of thread t at
// sm[q * blockDim.x + t].
enum ElasCoef { EC_F = 0, EC_G = 6, EC_MU = 12, EC_LAM = 18, EC_DIAG = 24, EC_COUNT = 27 };

// component A of the operator on the neighbours' x (elas_row64 with the coefficients at hand):
// face values +d at EC_F + 2 d, -d at EC_F + 2 d + 1, node values of mu and lambda alike
template <int A>
__device__ __forceinline__ double row_small(const Geo& G, const Nbr& nb, int c, const double* k,
                                            int ld, const double* const x[3]) {
  constexpr int D[2] = {(A + 1) % 3, (A + 2) % 3};
  auto co = [&](int q) { return k[q * ld]; };
  double v = co(EC_DIAG + A) * x[A][c];
  v = fma(-co(EC_F + 2 * A), x[A][at1<A>(nb, 1)], v);
  v = fma(-co(EC_F + 2 * A + 1), x[A][at1<A>(nb, -1)], v);
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int d = D[e];
    const int xp = d == 0 ? at1<0>(nb, 1) : (d == 1 ? at1<1>(nb, 1) : at1<2>(nb, 1));
    const int xm = d == 0 ? at1<0>(nb, -1) : (d == 1 ? at1<1>(nb, -1) : at1<2>(nb, -1));
    v = fma(-co(EC_G + 2 * d), x[A][xp], v);
    v = fma(-co(EC_G + 2 * d + 1), x[A][xm], v);
  }
  auto mixed = [&](auto dd) {
    constexpr int d = decltype(dd)::value;
    const double epp = x[d][at2<A, d>(nb, +1, +1)], epm = x[d][at2<A, d>(nb, -1, +1)];
    const double emp = x[d][at2<A, d>(nb, +1, -1)], emm = x[d][at2<A, d>(nb, -1, -1)];
    double m = co(EC_MU + 2 * d) * (epp - epm);
    m = fma(-co(EC_MU + 2 * d + 1), emp - emm, m);
    m = fma(co(EC_LAM + 2 * A), epp - emp, m);
    m = fma(-co(EC_LAM + 2 * A + 1), epm - emm, m);
    v = fma(-G.s_cross[A][d], m, v);
  };
  mixed(std::integral_constant<int, D[0]>{});
  mixed(std::integral_constant<int, D[1]>{});
  return v;
}

// The elasticity solve A du = r (E.r, E.p = D^{-1} r and the scalars E.S from k_elas_init):
// the increments in E.du, the scalars as the many-kernel form leaves them.  E.p carries z.
__global__ void __launch_bounds__(CGS_MAX_THREADS, 1) k_elas_cg(Geo G, Elas E,
                                                                unsigned int* words,
                                                                unsigned long long wait_ns) {
  extern __shared__ double coef[];
  __shared__ double sc[2];   // alpha, beta
  __shared__ CgScal sS;
  if (threadIdx.x == 0) sS = *E.S;
  __syncthreads();
  if (sS.status != CG_RUNNING) return;   // the same in every block: E.S is written at the end
  const int n = (int)G.nvox, c = blockIdx.x * blockDim.x + threadIdx.x, ld = blockDim.x;
  const bool on = c < n;
  const int i = on ? c % G.nx : 0, j = on ? (c / G.nx) % G.ny : 0, k = on ? c / (G.nx * G.ny) : 0;
  const Nbr nb = make_nbr(G, i, j, k);
  double* const kc = coef + threadIdx.x;   // this thread's coefficients: no other reads them
  if (on) {
    const int np[3] = {nb.at(1, 0, 0), nb.at(0, 1, 0), nb.at(0, 0, 1)};
    const int nm[3] = {nb.at(-1, 0, 0), nb.at(0, -1, 0), nb.at(0, 0, -1)};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      kc[(EC_F + 2 * d) * ld] = E.F[d][c];
      kc[(EC_F + 2 * d + 1) * ld] = E.F[d][nm[d]];
      kc[(EC_G + 2 * d) * ld] = E.G[d][c];
      kc[(EC_G + 2 * d + 1) * ld] = E.G[d][nm[d]];
      kc[(EC_MU + 2 * d) * ld] = E.mu[np[d]];
      kc[(EC_MU + 2 * d + 1) * ld] = E.mu[nm[d]];
      kc[(EC_LAM + 2 * d) * ld] = E.lam[np[d]];
      kc[(EC_LAM + 2 * d + 1) * ld] = E.lam[nm[d]];
      kc[(EC_DIAG + d) * ld] = E.dsum[d][c];
    }
  }
  double du[3] = {0.0, 0.0, 0.0}, r[3], p[3], q[3], dinv[3], z[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[a] = on ? E.r[a][c] : 0.0;
    z[a] = on ? E.p[a][c] : 0.0;
    dinv[a] = on ? E.dinv[a][c] : 0.0;
    p[a] = q[a] = 0.0;
  }
  double* const part_pq = E.q[0];   // A p stays in registers: its array holds the partials,
  double* const part_r = E.q[0] + gridDim.x;   // <p, q>, <r, D^{-1} r>, <r, r>
  unsigned int round = 0;
  double beta = 0.0;
  bool waited = true;
  for (;;) {
    double acc1[1] = {0.0};
    if (on) {
      // z as the neighbours left it: plain loads, which the wait's acquire made coherent (this
      // kernel writes the array, so they never take the read-only path)
      const double* const x[3] = {E.p[0], E.p[1], E.p[2]};
      const double w[3] = {row_small<0>(G, nb, c, kc, ld, x), row_small<1>(G, nb, c, kc, ld, x),
                           row_small<2>(G, nb, c, kc, ld, x)};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        p[a] = fma(beta, p[a], z[a]);   // the first time z and A z: p = q = beta = 0
        q[a] = fma(beta, q[a], w[a]);
        acc1[0] = fma(p[a], q[a], acc1[0]);
      }
    }
    leave_partials<1>(acc1, part_pq);
    if (!(waited = grid_wait(words, ++round, wait_ns))) break;
    if (threadIdx.x < 32) {
      const double pq = all_partials(part_pq);
      if (threadIdx.x == 0) {
        sS.pq = pq;
        sS.alpha = sS.rz / pq;
        sc[0] = sS.alpha;
      }
    }
    __syncthreads();
    const double alpha = sc[0];
    double acc2[2] = {0.0, 0.0};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      du[a] = fma(alpha, p[a], du[a]);
      r[a] = fma(-alpha, q[a], r[a]);
      z[a] = dinv[a] * r[a];
      if (on) E.p[a][c] = z[a];   // every block has applied its operator to the old z
      acc2[0] = fma(r[a], z[a], acc2[0]);
      acc2[1] = fma(r[a], r[a], acc2[1]);
    }
    leave_partials<2>(acc2, part_r);
    if (!(waited = grid_wait(words, ++round, wait_ns))) break;
    if (threadIdx.x < 32) {
      const double rz = all_partials(part_r), rr = all_partials(part_r + gridDim.x);
      if (threadIdx.x == 0) {
        cg_after_update(sS, rz, rr);
        sc[1] = sS.beta;
      }
    }
    __syncthreads();
    if (sS.status != CG_RUNNING) break;   // decided alike in every block
    beta = sc[1];
  }
  if (!waited) {
    if (threadIdx.x == 0) E.S->status = CG_TIMEOUT;
    return;
  }
  if (on) {
#pragma unroll
    for (int a = 0; a < 3; ++a) E.du[a][c] = du[a];
  }
  if (threadIdx.x == 0 && leave_last(words, gridDim.x)) *E.S = sS;
}

// The three Crank-Nicolson solves (C.r, C.p = D^{-1} r and the scalars C.S from k_cn_init) the
// same way: the fields C.x updated in place, C.p carrying z.  A finished solve's vectors stand
// still while the others go on.
__global__ void __launch_bounds__(CGS_MAX_THREADS, 1) k_cn_cg(Geo G, Cn3 C,
                                                              unsigned int* words,
                                                              unsigned long long wait_ns) {
  __shared__ double sa[3], sb[3];
  __shared__ CgScal sS[3];
  if (threadIdx.x < 3) sS[threadIdx.x] = C.S[threadIdx.x];
  __syncthreads();
  bool act[3];
#pragma unroll
  for (int s = 0; s < 3; ++s) act[s] = sS[s].status == CG_RUNNING;
  if (!(act[0] || act[1] || act[2])) return;   // the same in every block
  const int n = (int)G.nvox, c = blockIdx.x * blockDim.x + threadIdx.x;
  const bool on = c < n;
  const int i = on ? c % G.nx : 0, j = on ? (c / G.nx) % G.ny : 0, k = on ? c / (G.nx * G.ny) : 0;
  const Nbr nb = make_nbr(G, i, j, k);
  const int np[3] = {nb.at(1, 0, 0), nb.at(0, 1, 0), nb.at(0, 0, 1)};
  const int nm[3] = {nb.at(-1, 0, 0), nb.at(0, -1, 0), nb.at(0, 0, -1)};
  double fp[3], fm[3], x[3], r[3], p[3], q[3], z[3], beta[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    fp[d] = on ? C.Kf[d][c] : 0.0;
    fm[d] = on ? C.Kf[d][nm[d]] : 0.0;
    const bool go = on && act[d];
    x[d] = go ? C.x[d][c] : 0.0;
    r[d] = go ? C.r[d][c] : 0.0;
    z[d] = go ? C.p[d][c] : 0.0;
    p[d] = q[d] = beta[d] = 0.0;
  }
  const double diag = on ? C.dsum[c] : 0.0, dinv = on ? C.dinv[c] : 0.0;
  double* const part_pq = C.q[0];   // the array of A p, which stays in registers, holds three
  double* const part_r = C.q[1];    // doubles per block, the next six (at least 32 voxels each)
  unsigned int round = 0;
  bool waited = true;
  for (;;) {
    double acc1[3] = {0.0, 0.0, 0.0};
    if (on) {
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        if (!act[s]) continue;
        const double* zs = C.p[s];   // plain loads (see k_elas_cg)
        double w = diag * z[s];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          w = fma(-fp[d], zs[np[d]], w);
          w = fma(-fm[d], zs[nm[d]], w);
        }
        p[s] = fma(beta[s], p[s], z[s]);
        q[s] = fma(beta[s], q[s], w);
        acc1[s] = p[s] * q[s];
      }
    }
    leave_partials<3>(acc1, part_pq);
    if (!(waited = grid_wait(words, ++round, wait_ns))) break;
    if (threadIdx.x < 32) {
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        if (!act[s]) continue;
        const double pq = all_partials(part_pq + s * gridDim.x);
        if (threadIdx.x == 0) {
          sS[s].pq = pq;
          sS[s].alpha = sS[s].rz / pq;
          sa[s] = sS[s].alpha;
        }
      }
    }
    __syncthreads();
    double acc2[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      if (!act[s]) continue;
      const double alpha = sa[s];
      x[s] = fma(alpha, p[s], x[s]);
      r[s] = fma(-alpha, q[s], r[s]);
      z[s] = dinv * r[s];
      if (on) C.p[s][c] = z[s];
      acc2[2 * s] = r[s] * z[s];
      acc2[2 * s + 1] = r[s] * r[s];
    }
    leave_partials<6>(acc2, part_r);
    if (!(waited = grid_wait(words, ++round, wait_ns))) break;
    if (threadIdx.x < 32) {
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        if (!act[s]) continue;
        const double rz = all_partials(part_r + (2 * s) * gridDim.x);
        const double rr = all_partials(part_r + (2 * s + 1) * gridDim.x);
        if (threadIdx.x == 0) {
          cg_after_update(sS[s], rz, rr);
          sb[s] = sS[s].beta;
        }
      }
    }
    __syncthreads();
    bool any = false;   // decided alike in every block
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      if (!act[s]) continue;
      act[s] = sS[s].status == CG_RUNNING;
      beta[s] = sb[s];
      any |= act[s];
      if (on && !act[s]) C.x[s][c] = x[s];
    }
    if (!any) break;
  }
  if (!waited) {
    if (threadIdx.x < 3) C.S[threadIdx.x].status = CG_TIMEOUT;
    return;
  }
  if (threadIdx.x == 0 && leave_last(words, gridDim.x)) {
#pragma unroll
    for (int s = 0; s < 3; ++s) C.S[s] = sS[s];
  }
}

template <class View>
cudaError_t launch_small(void (*kernel)(Geo, View, unsigned int*, unsigned long long), const Geo& G,
                         const View& V, int doubles_per_thread, int sms, unsigned int* words,
                         unsigned long long wait_ns, cudaStream_t st) {
  const long long warps = (G.nvox + 31) / 32;
  const int threads = (int)(32 * ((warps + sms - 1) / sms));
  const int blocks = (int)((G.nvox + threads - 1) / threads);
  // the partials: up to six doubles per block in an array of one double per voxel
  if (threads > CGS_MAX_THREADS || 6LL * blocks > G.nvox) return cudaErrorInvalidValue;
  const size_t smem = (size_t)doubles_per_thread * threads * sizeof(double);
  if (smem > 32 * 1024) {   // the default 48 KB hold the static arrays too; a limit of the
                            // kernel, not of one launch: the most it ever takes
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             doubles_per_thread * CGS_MAX_THREADS * (int)sizeof(double));
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, G, V, words, wait_ns);
}

}  // namespace

// words: two zeroed words (tg_wait.cuh), left at zero by a launch that ended well
cudaError_t launch_elas_cg_small(const Geo& G, const Elas& E, int sms, unsigned int* words,
                                 unsigned long long wait_ns, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  TG_TIMED(K_ELAS_CG, st, e = launch_small(k_elas_cg, G, E, EC_COUNT, sms, words, wait_ns, st));
  return e;
}

cudaError_t launch_cn_cg_small(const Geo& G, const Cn3& C, int sms, unsigned int* words,
                               unsigned long long wait_ns, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  TG_TIMED(K_CN_CG, st, e = launch_small(k_cn_cg, G, C, 0, sms, words, wait_ns, st));
  return e;
}

}  // namespace tg
