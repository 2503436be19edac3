// tg_drive.h -- host-side decisions of the CG solves, free of CUDA so that the CPU tests build
// them too.
#pragma once

#include <algorithm>
#include <cmath>

namespace tg {

constexpr int CGS_MAX_THREADS = 512;   // most voxels per SM of a one-launch solve (tg_cg_small.cu)

// Whether an FP64 Jacobi solve on nvox voxels runs as one cooperative launch.  It needs every SM's
// registers for at most 512 voxels each.  sharers: the host threads that step simulations side
// by side (a concurrent batch), 1 alone.  The launch spends its waits idle, which the other
// members' solves fill only while several fit an SM; the queued kernels interleave at any size.
// So with sharers the solves in flight may take twice the chip's 512 voxels per SM.  ms for two
// steps of every member, queued -> one launch: 8 x 24^3 4.2 -> 4.0, 8 x 28^3 6.2 -> 6.9, 8 x 32^3
// 8.5 -> 11.3, 4 x 32^3 5.6 -> 5.6, 4 x 40^3 13.8 -> 14.6, 2 x 42^3 10.5 -> 8.6.
inline bool cg_small_fits(long long nvox, int sms, int sharers) {
  const long long most = (long long)CGS_MAX_THREADS * sms;
  return nvox <= most && (sharers <= 1 || nvox * sharers <= 2 * most);
}

// Blocks of one component (solve) of the flat FP64 vector updates, `want` to have one voxel pair
// per thread: two per SM, and never more than the partial-sum buffer holds (nine doubles for each
// of the nblocks of the grid-shaped kernels; three components leave two each).
inline long long flat_blocks(long long want, long long nblocks, int sms) {
  return std::max(1LL, std::min(want, std::min(2LL * sms, nblocks)));
}

// a launch that leaves the SMs fewer than four blocks each
inline bool few_blocks(long long blocks, int sms) { return blocks < 4LL * sms; }

// Planes a block of the FP32 operator marches, zc those of a grid-shaped launch of nblocks.  A
// block stages two planes more than it computes, so at one or a few planes per block (grids of
// 64^3 to 128^3, where 16 blocks per SM leave no more) a third to two thirds of the staging is
// halo: two chunks of planes per block where the launch still has four blocks per SM.  ms for two
// mixed steps, one -> two chunks: 64^3 12.9 -> 12.4, 128^3 15.5 -> 15.2; three or four chunks, or
// one wave of blocks, gain no more.  From nine planes a chunk on (256^3: 27) the halo is small and
// the blocks' number counts.
inline int op_planes(int zc, long long nblocks, int sms) {
  return zc <= 8 && !few_blocks(nblocks, sms) ? 2 * zc : zc;
}

// Iterations queued before the first look at a solve's flags, prev those of the last such solve.
inline int first_chunk(int prev) { return prev > 0 ? std::max(1, prev - prev / 8) : 4; }

// Iterations the running solves still need (S: the solves' scalars; `running` their status while
// they iterate; `grown` where a residual shows no rate).  Each read of the flags leaves the GPU
// idle for some 10 us, so the queue is filled by an estimate and not by a growing guess: a solve
// of 50 iterations takes two or three reads instead of four or five.  The residual is taken to
// keep falling at its mean rate from |rhs|, which is where a solve from zero starts (a refined
// one).  A solve from a good guess starts lower, and that rate comes out too high: from the second
// read on the rate since the first (first: the scalars read then, else null) counts too, for at
// most twice the iterations that it was seen over, as a few iterations' rate may be off.
template <class S>
int next_chunk(const S* host, const S* first, int nsolves, int running, int grown) {
  double need = 0.0;
  for (int r = 0; r < nsolves; ++r) {
    const S& s = host[r];
    if (s.status != running) continue;
    const double target = s.rtol * s.rtol * s.bb;
    if (!(s.it > 0 && target > 0.0 && s.rr > target && s.rr < s.bb)) return grown;
    const double left = std::log(s.rr / target);
    need = std::max(need, s.it * left / std::log(s.bb / s.rr));
    if (first && s.it > first[r].it && s.rr < first[r].rr) {
      const double seen = s.it - first[r].it;
      need = std::max(need, seen * std::min(left / std::log(first[r].rr / s.rr), 2.0));
    }
  }
  return (int)std::max(1.0, std::min(std::ceil(need), 64.0));
}

// The CUDA runtime's errors for a cooperative launch that it does not take, before anything ran:
// its blocks cannot all be resident (a process or partition that may use fewer SMs than the
// device has), or the device has no such launches.  cudaErrorCooperativeLaunchTooLarge and
// cudaErrorNotSupported; tg_api.cu asserts the values.
constexpr int COOP_REFUSED[2] = {720, 801};

enum SmallRun { SMALL_TAKEN, SMALL_QUEUE, SMALL_FAILED };

// Runs launch() (0 or the CUDA error) for a solve that fits one launch.  SMALL_QUEUE: the solve
// goes to the queued kernels, now and, with `refused` set, for the context's later solves.
template <class Launch>
SmallRun run_small(bool fits, bool& refused, Launch launch) {
  if (!fits || refused) return SMALL_QUEUE;
  const int e = launch();
  if (e == 0) return SMALL_TAKEN;
  refused = e == COOP_REFUSED[0] || e == COOP_REFUSED[1];
  return refused ? SMALL_QUEUE : SMALL_FAILED;
}

}  // namespace tg
