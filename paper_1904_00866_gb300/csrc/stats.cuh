// Fused per-step diagnostics: per-thread accumulation, warp-shuffle and
// shared-memory block reduction into one row of partials per block, then a
// single-block finish kernel that sums the rows in a fixed order (the result
// does not depend on scheduling).
#pragma once
#include <math.h>

#include "node_fp64.cuh"

namespace elbm {

// First statement of every kernel that launch_chained launches: lets the
// next kernel of the chain be scheduled as soon as every block of this one
// runs, and waits until the previous kernel has completed (no wait when the
// launch was not chained).  All threads call it before any access to memory
// another kernel writes, so completion is transitive along the chain.
// A chained grid may be resident while its predecessor still writes, so
// nothing the predecessor writes is constant for the kernel's duration: no
// __restrict__ and no read-only load on such data, which would let loads
// take the non-coherent path or move above the wait.
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Partial slots.  Slots [0, S_NSUM) are sums, the rest min / max.
enum {
  S_DRHO = 0,   // sum (rho - rho0)
  S_J0, S_J1, S_J2,
  S_KE,         // 1/2 sum |j|^2 / rho
  S_ASUM,
  S_H,          // sum H(f)      (CHECK)
  S_NODES,
  S_ACC2, S_ACCSTAR, S_FORMULA, S_BAND, S_FAR, S_DEGEN,
  S_ITERS, S_CAP, S_NOROOT,
  S_VIOL, S_MISMATCH,  // (CHECK)
  S_NSUM,
  S_AMIN = S_NSUM,
  S_AMAX,
  S_ADEV,       // max |alpha - alpha_FP64|   (CHECK)
  NSTAT
};

struct Acc {
  double drho, j0, j1, j2, ke, asum, h;
  double amin, amax, adev;
  unsigned nodes, acc2, accstar, formula, band, far, degen, iters, cap,
      noroot, viol, mismatch;

  __device__ __forceinline__ void init() {
    drho = j0 = j1 = j2 = ke = asum = h = 0.0;
    amin = INFINITY;
    amax = -INFINITY;
    adev = 0.0;
    nodes = acc2 = accstar = formula = band = far = degen = iters = cap =
        noroot = viol = mismatch = 0u;
  }
  __device__ __forceinline__ void add_moments(double dr, const double* j,
                                              double rho) {
    drho += dr;
    j0 += j[0];
    j1 += j[1];
    j2 += j[2];
    ke += 0.5 * (j[0] * j[0] + j[1] * j[1] + j[2] * j[2]) / rho;
  }
  __device__ __forceinline__ void add_moments_ke(double dr, const double* j,
                                                 double e) {
    drho += dr;
    j0 += j[0];
    j1 += j[1];
    j2 += j[2];
    ke += e;
  }
  __device__ __forceinline__ void add_alpha(double a, unsigned flags, int it) {
    nodes += 1;
    asum += a;
    amin = fmin(amin, a);
    amax = fmax(amax, a);
    acc2 += (flags & NF_ACCEPT_TWO) != 0;
    accstar += (flags & NF_ACCEPT_STAR) != 0;
    formula += (flags & NF_FORMULA) != 0;
    band += (flags & NF_BAND) != 0;
    degen += (flags & NF_DEGENERATE) != 0;
    cap += (flags & NF_ROOT_CAP) != 0;
    noroot += (flags & NF_NO_ROOT) != 0;
    iters += (unsigned)it;
  }
  __device__ __forceinline__ void add_check(double hf, bool v, bool mis,
                                            double dev) {
    h += hf;
    viol += v;
    mismatch += mis;
    adev = fmax(adev, dev);
  }

  // Reduce over the block and write partials[blockIdx.x * NSTAT + k].
  // Must be reached by every thread of the block.
  //
  // Bound by the FP64 pipe (64 cycles per warp addition): the seven FP64
  // sums are reduced together by halving the set at each exchange (lane
  // bits 16, 8, 4 pick the sum a lane keeps), 9 additions per warp instead
  // of 5 per sum; counters add as integers (warp reductions) and the alpha
  // extrema, positive or +-inf, order as integers.  A one-warp block of the
  // 64^2 FP64 step issues 95 FP64 instructions with its statistics, 201
  // with one butterfly per slot (14 -> 10 us in the same kernel).
  __device__ __forceinline__ void block_reduce_store(double* partials) {
    __shared__ double sm[32][NSTAT];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    constexpr int kFirst[8] = {S_DRHO, S_J0, S_J1, S_J2,
                               S_KE,   S_ASUM, S_H, S_H};
    {
      double v[8] = {drho, j0, j1, j2, ke, asum, h, 0.0};
#pragma unroll
      for (int half = 4, o = 16; half >= 1; half >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < half; ++k) {
          const double send = up ? v[k] : v[k + half];
          const double keep = up ? v[k + half] : v[k];
          v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      double t = v[0];
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      // lane bits 16, 8, 4: the sum's index
      const int k = (lane >> 2) & 7;
      int slot = kFirst[0];
#pragma unroll
      for (int q = 1; q < 7; ++q) slot = k == q ? kFirst[q] : slot;
      if ((lane & 3) == 0 && k < 7) sm[warp][slot] = t;
    }
    auto count = [&](int k, unsigned c) {
      const unsigned t = __reduce_add_sync(0xffffffffu, c);
      if (lane == 0) sm[warp][k] = (double)t;
    };
    count(S_NODES, nodes);
    count(S_ACC2, acc2);
    count(S_ACCSTAR, accstar);
    count(S_FORMULA, formula);
    count(S_BAND, band);
    count(S_FAR, far);
    count(S_DEGEN, degen);
    count(S_ITERS, iters);
    count(S_CAP, cap);
    count(S_NOROOT, noroot);
    count(S_VIOL, viol);
    count(S_MISMATCH, mismatch);
    // the extrema order as integers: alphas and deviations are >= 0, and
    // the empty maximum -inf (a negative integer) stays below them
    auto extreme = [&](int k, double v) {
      long long b = __double_as_longlong(v);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long w = __shfl_xor_sync(0xffffffffu, b, o);
        b = k == S_AMIN ? min(b, w) : max(b, w);
      }
      if (lane == 0) sm[warp][k] = __longlong_as_double(b);
    };
    extreme(S_AMIN, amin);
    extreme(S_AMAX, amax);
    extreme(S_ADEV, adev);
    __syncthreads();
    if (threadIdx.x < NSTAT) {
      const int k = threadIdx.x;
      double v = sm[0][k];
      for (int w = 1; w < nw; ++w) {
        const double x = sm[w][k];
        v = k < S_NSUM ? v + x : (k == S_AMIN ? fmin(v, x) : fmax(v, x));
      }
      partials[(long long)blockIdx.x * NSTAT + k] = v;
    }
  }
};

}  // namespace elbm
