// Batched heat step: many independent 2-D problems of uneven sizes advanced
// by ONE persistent, cooperative kernel per time step.
//
// The kernel walks the phases of a 3-stage SSP Runge-Kutta step:
//   for each stage: [x sweeps of every problem] -> [y sweeps] -> [FP64 update]
// and separates the phases with a grid barrier.  Within a sweep phase the CTAs
// take (problem, line tile) work items round-robin; every problem brings its
// own tile shape (points per lane E, warps per line, lines per tile), chosen
// per size class by the host-side autotuner.  Every wait is bounded: a grid
// barrier that does not complete within the wait limit records ST_TIMEOUT and
// the kernel returns.  Data written earlier in the same launch is read after a
// grid barrier, whose fences order it: the update and the accumulators through
// L2, the sweeps' lines by cp.async (through L1, which the fences invalidate).
#pragma once

#include "sweep.cuh"
#include "sweep_tma.cuh"

namespace molt {

struct alignas(16) BatchSweep {
  SweepArgs a;       // geometry, coefficients and tile shape of one (problem, axis)
  int E;             // points per lane (4, 8 or 16)
  int first_item;    // first work item of this problem in the phase
  int ntiles;
};

struct BatchUpdate {
  const float* acc;  // S of x
  const float* accy; // S of y
  double* u;         // u^n
  double* st1;       // stage states
  double* st2;
  float* copy;       // FP32 copy the sweeps read
  long long total;
  long long first_chunk;
};

struct BatchParams {
  int nprob;
  const BatchSweep* sweeps;   // [nprob][2]
  int items[2];               // work items of the x and y sweep phases
  const BatchUpdate* updates; // [nprob]
  long long chunks;           // work items of the update phase
  double coefS;               // -beta^2
  int stages;                 // 3 (a full step) or 1 (tuning)
  int phase_mask;             // bit 0: x sweeps, bit 1: y sweeps, bit 2: updates
  unsigned int* bar_count;
  unsigned int* bar_gen;
  int* status;
  long long wait_limit;       // cycles
  int skip_arrive;            // test hook: CTA 0 never arrives at the first barrier
  unsigned int buf_bytes;     // shared bytes of one of the two tile buffers
};

constexpr size_t kBatchHead = 128;   // shared bytes of the warps' totals (16 warps)
static_assert(tile_head_bytes(1, 16, 4) <= kBatchHead, "totals of 16 warps");

// 4-byte asynchronous copy: the tile's values land in the padded layout of
// the compute core with no pass of their own.  (The inputs were written
// earlier in the launch by other CTAs; the grid barrier's fences order them.)
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  const unsigned int d = static_cast<unsigned int>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned int d = static_cast<unsigned int>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// points per update work item: two a thread (64 problems, 2 steps: 8 / 4 / 2 /
// 1 points a thread 11.1 / 10.8 / 10.6 / 10.8 ms, an L2 prefetch of the next
// item 0.2 ms slower)
constexpr int kChunk = 1024;

// Grid barrier with a bounded wait (cooperative launch: all CTAs resident).
__device__ __forceinline__ bool grid_sync(const BatchParams& p, bool skip) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned int* gen = p.bar_gen;
    const unsigned int g = *gen;
    __threadfence();
    bool done = false;
    if (!skip) {
      const unsigned int arrived = atomicAdd(p.bar_count, 1u) + 1u;
      if (arrived == gridDim.x) {
        *p.bar_count = 0u;
        __threadfence();
        atomicAdd(p.bar_gen, 1u);
        done = true;
      }
    }
    if (!done) {
      const long long t0 = clock64();
      while (*gen == g) {
        if (clock64() - t0 > p.wait_limit) {
          atomicOr(p.status, ST_TIMEOUT);
          ok = 0;
          break;
        }
        __nanosleep(128);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// Starts the copy of one (problem, line tile) work item into shared memory:
// its arguments and its lines.  The tile shape fills the CTA exactly (32 * nwl
// * W == blockDim.x) and the lines are an exact fit (n = 32*nwl*E).
__device__ __forceinline__ void batch_fetch(const BatchSweep& bs, BatchSweep* args, float* lines, long long item) {
  const SweepArgs& a = bs.a;
  const char* src = reinterpret_cast<const char*>(&bs);
  char* dst = reinterpret_cast<char*>(args);
  for (int c = threadIdx.x; c < int(sizeof(BatchSweep) / 16); c += blockDim.x) cp_async16(dst + 16 * c, src + 16 * c);
  const long long line0 = (item - bs.first_item) * a.W;
  const int warp = threadIdx.x >> 5, lw = warp / a.nwl;
  const int tl = (warp - lw * a.nwl) * 32 + (threadIdx.x & 31);
  const float* in = static_cast<const float*>(a.in);
  auto put = [](float* d, const float* g) { cp_async4(d, g); };
  if (bs.E == 16) load_tile<float, float, 16>(a, in, lines, line0, lw, tl, put);
  else if (bs.E == 8) load_tile<float, float, 8>(a, in, lines, line0, lw, tl, put);
  else load_tile<float, float, 4>(a, in, lines, line0, lw, tl, put);
  cp_async_commit();
}

template <int E>
__device__ __forceinline__ void batch_tile(const SweepArgs& a, const TileSmem& sm, long long line0) {
  const int lw = (threadIdx.x >> 5) / a.nwl;
  compute_lines<float, JQ_D0, false, E>(a, sm, line0 + lw < a.g.nlines);
  epilogue_tile<float, double, EPI_ACC_SET, E, true>(a, static_cast<const float*>(sm.lines), line0, 0.0);
}

// Problem of a work item, by one warp (the items of problem k start at
// first_item): lanes compare 32 problems at a time.
__device__ __forceinline__ int find_problem(const BatchParams& p, long long item, int ax, int lane) {
  int count = 0;
  for (int k0 = 0; k0 < p.nprob; k0 += 32) {
    const int k = k0 + lane;
    const bool le = k < p.nprob && p.sweeps[k * 2 + ax].first_item <= item;
    count += __popc(__ballot_sync(0xffffffffu, le));
  }
  return count - 1;
}

// Compiled for two CTAs per SM (64 registers; more spills than at 128, but
// the second resident CTA covers the phases' memory latency: 64 problems, two
// steps, 1 / 2 / 3 CTAs per SM 14.1 / 11.4 / 15.0 ms, before the update's
// smaller chunks; 10.4 ms now).
#ifndef MOLT_BATCH_MIN_BLOCKS
#define MOLT_BATCH_MIN_BLOCKS 2
#endif
#ifndef MOLT_BATCH_KERNEL_TU
// defined in csrc/batch.cu (its own translation unit: FP32 <-> FP64
// conversions in place, MOLT_CONV_SELECT)
__global__ void batch_heat_kernel(const BatchParams p);
#else
__global__ void __launch_bounds__(512, MOLT_BATCH_MIN_BLOCKS) batch_heat_kernel(const BatchParams p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ BatchSweep sa[2];
  __shared__ int s_prob[3];   // problem of this item, the next and the one after (rotating)
  static const double rk[3][2] = {{0.0, 1.0}, {0.75, 0.25}, {1.0 / 3.0, 2.0 / 3.0}};
  const int lane = threadIdx.x & 31;
  float* buf[2] = {reinterpret_cast<float*>(smem_raw + kBatchHead),
                   reinterpret_cast<float*>(smem_raw + kBatchHead + p.buf_bytes)};
  bool first = true;
  for (int s = 0; s < p.stages; ++s) {
    for (int ax = 0; ax < 2; ++ax) {
      if (p.phase_mask & (1 << ax)) {
        // the CTA's items: while one is computed, the next one's lines and
        // arguments arrive in the other buffer and warp 0 looks up the
        // problem of the one after
        const long long step = gridDim.x;
        if (threadIdx.x < 32) {
          const int p0 = find_problem(p, blockIdx.x, ax, lane), p1 = find_problem(p, blockIdx.x + step, ax, lane);
          if (lane == 0) {
            s_prob[0] = p0;
            s_prob[1] = p1;
          }
        }
        __syncthreads();
        if (blockIdx.x < p.items[ax]) batch_fetch(p.sweeps[s_prob[0] * 2 + ax], &sa[0], buf[0], blockIdx.x);
        int cur = 0, slot = 0;
        for (long long item = blockIdx.x; item < p.items[ax]; item += step) {
          cp_async_wait_all();
          __syncthreads();   // the item is in place; the other buffer's readers are done
          const int s1 = slot == 2 ? 0 : slot + 1, s2 = s1 == 2 ? 0 : s1 + 1;
          if (item + step < p.items[ax])
            batch_fetch(p.sweeps[s_prob[s1] * 2 + ax], &sa[cur ^ 1], buf[cur ^ 1], item + step);
          if (threadIdx.x < 32) {
            const int p2 = find_problem(p, item + 2 * step, ax, lane);
            if (lane == 0) s_prob[s2] = p2;
          }
          const BatchSweep& bs = sa[cur];
          TileSmem sm{};
          sm.totals = smem_raw;
          sm.lines = buf[cur];
          const long long line0 = (item - bs.first_item) * bs.a.W;
          if (bs.E == 16) batch_tile<16>(bs.a, sm, line0);
          else if (bs.E == 8) batch_tile<8>(bs.a, sm, line0);
          else batch_tile<4>(bs.a, sm, line0);
          cur ^= 1;
          slot = s1;
        }
      }
      const bool skip = first && p.skip_arrive && blockIdx.x == 0;
      first = false;
      if (!grid_sync(p, skip)) return;
    }
    if (p.phase_mask & 4) {
      const double a0 = rk[s][0], a1 = rk[s][1];
      bool bad = false;
      // chunk c of all problems goes to CTA c mod gridDim.x
      for (int q = 0; q < p.nprob; ++q) {
        const BatchUpdate& U = p.updates[q];
        const long long rot = U.first_chunk % gridDim.x;
        const double* us = s == 0 ? U.u : (s == 1 ? U.st1 : U.st2);
        double* dstp = s == 0 ? U.st1 : (s == 1 ? U.st2 : U.u);
        for (long long i0 = ((blockIdx.x + gridDim.x - rot) % gridDim.x) * kChunk; i0 < U.total;
              i0 += (long long)gridDim.x * kChunk) {
          const long long i1 = i0 + kChunk < U.total ? i0 + kChunk : U.total;
          // (all loads of a thread's points are issued before its stores)
          constexpr int kPer = kChunk / 512;
          double uu[kPer], ss[kPer];
          float aa[kPer], ay[kPer];
#pragma unroll
          for (int k = 0; k < kPer; ++k) {
            const long long i = i0 + threadIdx.x + (long long)k * blockDim.x;
            if (i < i1) {
              ss[k] = __ldcg(us + i);
              uu[k] = s == 0 ? 0.0 : __ldcg(U.u + i);
              aa[k] = __ldcg(U.acc + i);
              ay[k] = __ldcg(U.accy + i);
            }
          }
#pragma unroll
          for (int k = 0; k < kPer; ++k) {
            const long long i = i0 + threadIdx.x + (long long)k * blockDim.x;
            if (i < i1) {
              // the axis sums meet in FP64: no FP32 rounding at their joint size
              const double t = fma(p.coefS, f2d(aa[k]), fma(p.coefS, f2d(ay[k]), ss[k]));
              const double r = s == 0 ? t : fma(a0, uu[k], a1 * t);
              dstp[i] = r;
              U.copy[i] = d2f(r);
              bad |= nonfinite(r);
            }
          }
        }
      }
      if (bad) atomicOr(p.status, ST_NONFINITE);
      if (s + 1 < p.stages && !grid_sync(p, false)) return;
    }
  }
}

#endif  // MOLT_BATCH_KERNEL_TU

}  // namespace molt
