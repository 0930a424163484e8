// The grid barrier of the resident sweeps and the warp that runs it: one launch
// does every sweep of an inner solve, one bounded barrier per sweep.
//
// The barrier is one 64-bit word.  Low half: arrivals.  High half: the decision,
// (flag << 28) | the sweep it was made in (a CTA that reads the word late must not
// act on the next sweep's decision); bit 63: a wait ran out.
// The residual terms of sweep k - 1 are formed by the other warps while barrier k
// is awaited and left in part[k & 1]; the CTA's sum is out with barrier k + 1, CTA
// 0 closes it in sweep k + 2, and the decision ends every CTA before sweep k + 3.
#pragma once

#include <cstdint>

#include "vtm_internal.h"

namespace vtm {

// What the word can count: 32 bits of arrivals (half of them used, so that no carry
// reaches the decision), 28 bits of sweep number.
inline bool res_counts(int budget, int ctas) { return (int64_t)budget * ctas < (1ll << 31) && budget < (1 << 27); }

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// fixed-order sum of the warps' partials (one warp, valid in lane 0)
__device__ __forceinline__ double res_sum(const double* part, int count, int lane) {
  double v = lane < count ? part[lane] : 0.0;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// The residual rule of sweep_decide with its state in the deciding thread.
struct ResDecision {
  double tol2, bnorm2, first, best, last;
  int k_max, stall, best_k, conv;
  __device__ void load(const SweepCtrl* c) {
    tol2 = c->tol2;
    bnorm2 = c->bnorm2;
    first = best = last = 0.0;
    k_max = c->k_max;
    stall = c->stall;
    best_k = conv = 0;
  }
  __device__ int close(int k, double tot, double* hist, int hist_len) {
    int flag = 0;
    if (k > 1) {
      const int ks = k - 1;
      if (hist && ks <= hist_len) hist[ks - 1] = sqrt(tot / bnorm2);
      if (ks == 1) first = tot;
      last = tot;
      if (ks == 1 || tot < 0.81 * best) {
        best = tot;
        best_k = ks;
      }
      if (!isfinite(tot) || (ks > 1 && tot > 1e12 * first && first > 0)) {
        flag = 3;
      } else if (tot <= tol2) {
        flag = 1;
        conv = ks;
      } else if (stall > 0 && ks - best_k >= stall) {
        flag = 4;
        conv = ks;
      }
    }
    if (!flag && k >= k_max) flag = 2;
    return flag;
  }
  __device__ void store(SweepCtrl* c, int k, int flag) const {
    c->k = k + 1;
    c->conv_sweep = conv;
    c->best_k = best_k;
    c->best_res2 = best;
    c->first_res2 = first;
    c->last_res2 = last;
    c->flag = flag;
  }
};

// The control warp of a CTA with nw other warps (all of them meet its two CTA
// barriers per sweep).  s_part: [2][stride] residual partials of the warps.
__device__ __forceinline__ void res_control(SweepCtrl* ctrl, unsigned long long* bar, double* part, double* hist,
                                            int hist_len, uint32_t max_polls, int* s_flag, const double* s_part,
                                            int stride, int nw, int lane) {
  ResDecision dec;
  dec.load(ctrl);
  for (int k = 1;; ++k) {
    __syncthreads();  // the waves of sweep k - 1 are out and the flag is read
    if (*((volatile int*)s_flag)) break;
    int f = 0;
    if (k > 1) {
      const double v = res_sum(s_part + ((k - 1) & 1) * stride, nw, lane);
      if (lane == 0) part[(size_t)((k - 1) & 1) * gridDim.x + blockIdx.x] = v;
      if (blockIdx.x == 0 && k > 2) {  // the partials of sweep k - 2 came with barrier k - 1
        const double* pk = part + (size_t)(k & 1) * gridDim.x;
        double t = 0.0;
        for (int i = lane; i < (int)gridDim.x; i += 32) t += __ldcg(pk + i);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0 && (f = dec.close(k - 2, t, hist, hist_len))) dec.store(ctrl, k - 2, f);
      }
    }
    __syncthreads();  // every wave of sweep k is written
    if (lane == 0) {
      if (f) atomicAdd(bar, (unsigned long long)((uint32_t)f << 28 | (uint32_t)k) << 32);
      __threadfence();  // the CTA's waves and partial before its arrival
      atomicAdd(bar, 1ull);
      const unsigned need = (unsigned)k * gridDim.x;
      uint32_t i = 0;
      unsigned long long w;
      while (true) {
        w = ld_acquire_u64(bar);
        if ((unsigned)w >= need || (w >> 63)) break;
        if (++i >= max_polls) {  // give up; the word tells every CTA still waiting
          atomicCAS(&ctrl->flag, 0, 5);
          atomicOr(bar, 1ull << 63);
          w = 1ull << 63;
          break;
        }
      }
      if (w >> 63) *((volatile int*)s_flag) = 5;
      else if ((uint32_t)(w >> 32) && (int)((w >> 32) & 0x0fffffffu) == k) *((volatile int*)s_flag) = (int)(w >> 60);
    }
  }
}

}  // namespace vtm
