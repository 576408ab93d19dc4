// Stream-collide kernel in FP64 arithmetic: FP64 storage with every alpha
// mode, FP32 / FP16 storage with ROOT and SECANT.
//
// A thread collides one node per iteration, consecutive threads consecutive
// nodes of the flat index (ragged rows leave no lane idle).  Nodes near
// equilibrium take the series path (series64.cuh: ~120 FP64 instructions
// per D3Q27 FORMULA node and 60 per D2Q9 node, at 64 cycles each the
// kernel's bound: FP64 pipe 84 % busy for D2Q9, about 60 % for D3Q27, whose
// FP32 and integer part does not overlap with it at two warps per scheduler).
// The others take the logarithm path (node_fp64.cuh) out of line, so that its
// registers do not count here: each warp collects them in shared memory and
// runs them 32 at a time, one per lane, from their stored values.
//
// Measured (GB300, us per step; before: every node through the logarithm
// path, one row segment of 32 nodes per warp, ~700 FP64 instructions per
// D2Q9 FORMULA node):
//   D2Q9 1024^2 shear layer, FP64 storage, FORMULA     1326 ->  128
//   D2Q9 1024^2 shear layer, FP32 storage, ROOT       11560 ->  565
//   D3Q27 128^3 Taylor-Green, FP64 storage, FORMULA    7960 ->  667
//   D2Q9 64^2, FP64 storage, FORMULA with statistics     69 ->   10
// One FORMULA step with a share of the nodes at |x| ~ 0.2, all through the
// logarithm path -> each warp's far nodes where it meets them -> collected:
//   D3Q27 96^3    1 %  6449 -> 3574 ->  509     D2Q9 1024^2  1504 ->  752 ->  274
//                10 %  7026 -> 9142 -> 1437                  1824 -> 1842 ->  447
//               100 %  5481 -> 6291 -> 5975                  2039 -> 2169 -> 2084
// (a state with every node far pays for the attempt, and with ROOT for the 12
// warps per SM: D2Q9 43.7 -> 46.8 ms; the first step after initialisation,
// all by logarithms, takes what it took).
// Populations after 8 to 54 steps are as far from the 64-bit reference as
// before or nearer (1.3e-15 against 1.4e-15 on 128^3).
#pragma once
#include "fp16_storage.cuh"
#include "sc32.cuh"
#include "series64.cuh"
#include "stats.cuh"
#include "stream_collide.cuh"

namespace elbm {

// What the statistics need of one collided node.
struct Collided64 {
  double rho, j[3], alpha;
  unsigned flags;
  int iters;
};

// The populations of a node from its stored values in f_in.
template <class L, class T>
__device__ __forceinline__ void gather64(const StepParams& p, unsigned node,
                                         double (&f)[L::Q]) {
  const T* fin = static_cast<const T*>(p.f_in);
  int x, y, z;
  node_xyz<L>(p, node, x, y, z);
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const T v = fin[(long long)i * p.ps + src_index<L>(p, i, x, y, z)];
    if constexpr (sizeof(T) == 8)
      f[i] = v;
    else if constexpr (sizeof(T) == 2)
      f[i] = h16_to_f<L>(v, i, p.rho0);
    else
      f[i] = p.unshifted ? (double)v : L::w(i) * p.rho0 + (double)v;
  }
}

// FP64 entropy check (Eq. (7)) of a node at the alpha it took, by either
// path; out of line, so that a checked step differs from the others in its
// statistics only.
template <class L, class T>
__device__ __noinline__ Check64 check64_at(const StepParams& p, unsigned node,
                                           double alpha) {
  Node64<L> nd;
  gather64<L, T>(p, node, nd.f);
  node64_prepare(nd);
  return node64_check(nd, alpha);
}

// The logarithm path of one node, from its stored values in f_in.  Flags
// NF_BAD_*: the state is invalid and the node is copied unchanged.
template <class L, class T, int MODE>
__device__ __noinline__ Collided64 far64_node(const StepParams& p,
                                              unsigned node) {
  T* fout = static_cast<T*>(p.f_out);
  Node64<L> nd;
  gather64<L, T>(p, node, nd.f);
  Collided64 r;
  r.iters = 0;
  r.alpha = 2.0;
  r.flags = node64_prepare(nd);
  r.rho = nd.rho;
  r.j[0] = nd.j[0];
  r.j[1] = nd.j[1];
  r.j[2] = nd.j[2];
  const bool bad = r.flags != 0;
  double ab = 0.0;
  if (!bad) {
    r.alpha = node64_alpha<L, MODE>(nd, p.secant_iters, r.flags, r.iters);
    if (sizeof(T) != 8) r.alpha = (double)__double2float_rd(r.alpha);
    ab = r.alpha * p.beta;
  } else {
    atomicOr(p.err_flags, r.flags);
  }
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const double val =
        bad ? nd.f[i] : fma(ab, nd.f[i] * nd.x[i], nd.f[i]);
    T& out = fout[(long long)i * p.ps + node];
    if constexpr (sizeof(T) == 8)
      out = val;
    else if constexpr (sizeof(T) == 2)
      out = h16_from_dev<L>(val - L::w(i) * p.rho0, i);
    else
      out = (T)(p.unshifted ? val : val - L::w(i) * p.rho0);
  }
  return r;
}

template <class L, class T, int MODE, int DIAG, int CHECK>
__global__ void __launch_bounds__(128) k_sc64(const StepParams p) {
  chain_begin();
  constexpr int Q = L::Q;
  const T* fin = static_cast<const T*>(p.f_in);
  T* fout = static_cast<T*>(p.f_out);
  Acc acc;
  if (DIAG) acc.init();
  auto check = [&](unsigned node, double alpha, unsigned flags) {
    const Check64 ck = check64_at<L, T>(p, node, alpha);
    acc.add_check(ck.h, ck.violation, decision_mismatch(flags, ck.accept_ref),
                  fabs(alpha - ck.alpha_ref));
  };
  // this warp's nodes for the logarithm path (warp-uniform count, below 32
  // before a round adds up to 32)
  __shared__ unsigned far_s[4][64];   // blocks of up to 128 threads
  unsigned* far = far_s[threadIdx.x >> 5];
  int nfar = 0;
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long k0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
       k0 < p.n || nfar > 0; k0 += stride) {
    const long long k = k0 + lane;
    const unsigned node = (unsigned)k;
    bool is_far = k < p.n;
    Near64<L> nd;
    if (k < p.n) {
      int x, y, z;
      node_xyz<L>(p, node, x, y, z);
      // element offsets of the neighbours along each axis
      const int dx[3] = {x == p.nx - 1 ? 1 - p.nx : 1, 0,
                         x == 0 ? p.nx - 1 : -1};
      const long long rx = p.nx, pl = (long long)p.nx * p.ny;
      const long long dy[3] = {y == p.ny - 1 ? rx * (1 - p.ny) : rx, 0,
                               y == 0 ? rx * (p.ny - 1) : -rx};
      const long long dz[3] = {z == p.nz - 1 ? pl * (1 - p.nz) : pl, 0,
                               z == 0 ? pl * (p.nz - 1) : -pl};
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const long long src = k + dx[L::c(i, 0) + 1] + dy[L::c(i, 1) + 1] +
                              (L::D == 3 ? dz[L::c(i, 2) + 1] : 0);
        nd.f[i] = load64<L, T>(fin[(long long)i * p.ps + src], i, p.rho0,
                               p.unshifted);
      }
    }
    Series64 se;
    if (is_far && near64_prepare(nd, se, sizeof(T) == 8 ? kSeriesXMax
                                                        : kSeriesXMaxRounded)) {
      is_far = false;
      unsigned flags = 0;
      int iters = 0;
      double alpha = 2.0;
      if (MODE == MODE_ROOT)
        alpha = alpha_root_near(nd, se, flags, iters);
      else if (MODE == MODE_SECANT)
        alpha = alpha_secant_near(se, p.secant_iters, flags, iters);
      else
        alpha = alpha_formula_near(se, flags);
      if (sizeof(T) != 8) alpha = (double)__double2float_rd(alpha);
      const double ab = alpha * p.beta;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const double val = fma(ab, nd.n[i], nd.f[i]);
        T& out = fout[(long long)i * p.ps + k];
        if constexpr (sizeof(T) == 8)
          out = val;
        else if constexpr (sizeof(T) == 2)
          out = h16_from_dev<L>(fma(-L::w(i), p.rho0, val), i);
        else
          out = (T)(p.unshifted ? val : fma(-L::w(i), p.rho0, val));
      }
      if (p.alpha_map) p.alpha_map[k] = (float)alpha;
      if (DIAG) {
        const double j[3] = {nd.j[0] * nd.unit, nd.j[1] * nd.unit,
                             L::D == 3 ? nd.j[2] * nd.unit : 0.0};
        // 1/2 rho |u|^2 with u = j / rho in the node's units
        const double ke = nd.unit * nd.inv_rho *
                          (nd.j[0] * nd.j[0] + nd.j[1] * nd.j[1] +
                           nd.j[2] * nd.j[2]);
        acc.add_moments_ke(fma(nd.rho, nd.unit, -p.rho0), j, 0.5 * ke);
        acc.add_alpha(alpha, flags, iters);
        if (CHECK) check(node, alpha, flags);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, is_far);
    if (is_far) far[nfar + __popc(m & ((1u << lane) - 1u))] = node;
    nfar += __popc(m);
    if (nfar >= 32 || (nfar > 0 && k0 + stride >= p.n)) {   // warp-uniform
      const int take = min(nfar, 32);
      nfar -= take;
      __syncwarp();
      const bool mine = lane < take;
      const unsigned fn = mine ? far[nfar + lane] : 0u;
      __syncwarp();
      if (mine) {
        const Collided64 c = far64_node<L, T, MODE>(p, fn);
        if (!(c.flags & (NF_BAD_NEG | NF_BAD_NONFINITE))) {
          if (p.alpha_map) p.alpha_map[fn] = (float)c.alpha;
          if (DIAG) {
            acc.add_moments(c.rho - p.rho0, c.j, c.rho);
            acc.add_alpha(c.alpha, c.flags, c.iters);
            if (CHECK) check(fn, c.alpha, c.flags);
          }
        }
      }
    }
  }
  if (DIAG) acc.block_reduce_store(p.partials);
}

}  // namespace elbm
