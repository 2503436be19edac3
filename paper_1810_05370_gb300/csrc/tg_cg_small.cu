// tg_cg_small.cu -- the FP64 Jacobi-CG solves of small grids as one launch each.
//
// On grids up to a few ten thousand voxels a CG iteration of the many-kernel form is latency:
// at 32^3 its three kernels carry 5 us of arithmetic and take 22 us, most of it launches,
// ramps and the last block's sum.  Here one cooperative kernel runs the whole solve.  Every
// thread owns one voxel and keeps the voxel's part of the CG vectors (increment, residual,
// direction, A p, inverse diagonal) in registers from the first iteration to the last; only
// the search direction goes through memory, for the neighbours' operator.  An iteration has
// three waits: two carry sums (each block leaves its partial sums before the wait and one warp
// of every block adds all of them after it, in block order, so every block takes the same
// decision with no second round trip), the third publishes the new direction.
//
// One block per SM: the grid is dealt out in blocks of 32 ceil(n / (32 SMs)) threads, which
// spreads the FP64 work (78 of the operator's operations per voxel, on a pipe of two lanes per
// clock and SM) evenly over the SMs; 512 threads of 128 registers fill an SM's register file,
// so grids up to 512 voxels per SM (77824 on 152 SMs) take this form.
//
// The waits are bounded in time: a block that gives up marks the solve CG_TIMEOUT and returns,
// and so do the others in their turn.  Launched cooperatively, so all blocks are resident.
#include <algorithm>

#include "tg_internal.cuh"

namespace tg {
namespace {

constexpr int CGS_MAX_THREADS = 512;
constexpr unsigned long long CGS_WAIT_NS = 2000000000ull;   // 2 s for a wait of microseconds

__device__ __forceinline__ unsigned long long timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Waits until all blocks of the launch have arrived for the round-th time (round = 1, 2, ...);
// everything any thread wrote before its block's arrival is visible after it.  False in every
// thread of the block if the wait ran out.
__device__ __forceinline__ bool grid_wait(unsigned int* arrived, unsigned int round) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int want = round * gridDim.x;
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrived) : "memory");
    int good = 1;
    unsigned long long t0 = 0;
    for (unsigned int spin = 0;; ++spin) {
      unsigned int seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(arrived) : "memory");
      if ((int)(seen - want) >= 0) break;   // rounds may wrap
      if ((spin & 255u) == 0u) {
        const unsigned long long t = timer_ns();
        if (t0 == 0) t0 = t;
        if (t - t0 > CGS_WAIT_NS) {
          good = 0;
          break;
        }
      }
    }
    __threadfence();
    ok = good;
  }
  __syncthreads();
  return ok != 0;
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

// Leaves the launch's two counters at zero for the next one: the last block out resets them.
__device__ __forceinline__ void leave_counters(unsigned int* counters) {
  if (threadIdx.x == 0 && ticket_acq_rel(counters + 1) == gridDim.x - 1) {
    counters[0] = 0u;
    counters[1] = 0u;
  }
}

// The elasticity solve A du = r (E.r, E.p = D^{-1} r and the scalars E.S from k_elas_init):
// the increments in E.du, the scalars as the many-kernel form leaves them.
__global__ void __launch_bounds__(CGS_MAX_THREADS, 1) k_elas_cg(Geo G, Elas E,
                                                                unsigned int* counters) {
  __shared__ double sc[2];   // alpha; then beta
  __shared__ CgScal sS;
  if (threadIdx.x == 0) sS = *E.S;
  __syncthreads();
  if (sS.status != CG_RUNNING) return;   // the same in every block: E.S is written at the end
  const int n = (int)G.nvox, c = blockIdx.x * blockDim.x + threadIdx.x;
  const bool on = c < n;
  const int i = on ? c % G.nx : 0, j = on ? (c / G.nx) % G.ny : 0, k = on ? c / (G.nx * G.ny) : 0;
  const Nbr nb = make_nbr(G, i, j, k);
  double du[3] = {0.0, 0.0, 0.0}, r[3], p[3], q[3], dinv[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[a] = on ? E.r[a][c] : 0.0;
    p[a] = on ? E.p[a][c] : 0.0;
    dinv[a] = on ? E.dinv[a][c] : 0.0;
    q[a] = 0.0;
  }
  double* const part_pq = E.q[0];   // A p stays in registers: its array holds the partials,
  double* const part_r = E.q[0] + gridDim.x;   // <p, q>, <r, D^{-1} r>, <r, r>
  unsigned int round = 0;
  bool waited = true;
  for (;;) {
    double acc1[1] = {0.0};
    if (on) {
      // the direction as the neighbours left it: plain loads, which the wait's acquire made
      // coherent (this kernel writes E.p, so they never take the read-only path)
      const double* const x[3] = {E.p[0], E.p[1], E.p[2]};
      q[0] = elas_row64<0>(G, nb, c, E, x);
      q[1] = elas_row64<1>(G, nb, c, E, x);
      q[2] = elas_row64<2>(G, nb, c, E, x);
      acc1[0] = fma(p[2], q[2], fma(p[1], q[1], p[0] * q[0]));
    }
    leave_partials<1>(acc1, part_pq);
    if (!(waited = grid_wait(counters, ++round))) break;
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
    double acc2[2] = {0.0, 0.0}, z[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      du[a] = fma(alpha, p[a], du[a]);
      r[a] = fma(-alpha, q[a], r[a]);
      z[a] = dinv[a] * r[a];
      acc2[0] = fma(r[a], z[a], acc2[0]);
      acc2[1] = fma(r[a], r[a], acc2[1]);
    }
    leave_partials<2>(acc2, part_r);
    if (!(waited = grid_wait(counters, ++round))) break;
    if (threadIdx.x < 32) {
      const double rz = all_partials(part_r), rr = all_partials(part_r + gridDim.x);
      if (threadIdx.x == 0) {
        cg_after_update(sS, rz, rr);
        sc[1] = sS.beta;
      }
    }
    __syncthreads();
    if (sS.status != CG_RUNNING) break;   // decided alike in every block
    const double beta = sc[1];
    if (on) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        p[a] = fma(beta, p[a], z[a]);
        E.p[a][c] = p[a];
      }
    }
    if (!(waited = grid_wait(counters, ++round))) break;
  }
  if (!waited) {   // the counters stay as they are: the context is unusable after a timeout
    if (threadIdx.x == 0) E.S->status = CG_TIMEOUT;
    return;
  }
  if (on) {
#pragma unroll
    for (int a = 0; a < 3; ++a) E.du[a][c] = du[a];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *E.S = sS;
  leave_counters(counters);
}

}  // namespace

bool cg_small_ok(const Geo& G, int sms) {
  return G.nvox <= (long long)CGS_MAX_THREADS * sms && sms > 0;
}

// counters: two zeroed words.  The partials (three doubles per block of at least 32 voxels,
// except the last) fit the array of A p, which holds a double per voxel, from 4 voxels on.
cudaError_t launch_elas_cg_small(const Geo& G, const Elas& E, int sms, unsigned int* counters,
                                 cudaStream_t st) {
  const long long warps = (G.nvox + 31) / 32;
  const int threads = (int)(32 * ((warps + sms - 1) / sms));
  const int blocks = (int)((G.nvox + threads - 1) / threads);
  if (threads > CGS_MAX_THREADS || 3LL * blocks > G.nvox) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  TG_TIMED(K_ELAS_CG, st, cudaLaunchKernelEx(&cfg, k_elas_cg, G, E, counters));
  return cudaGetLastError();
}

}  // namespace tg
