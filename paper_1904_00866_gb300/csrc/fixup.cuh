// Fixup kernels of the FP32 / FP16 FORMULA step, after the stream-collide
// kernel; both read f_in (unchanged during the step) and write f_out.
//   k_refine_stage: the second stage of the nodes whose FP32 entropy
//     decision was not certified (the stream-collide kernel wrote them with
//     the certified alpha and put their stored values in a buffer): f^eq - f
//     recomputed in double-float arithmetic, the decision retaken with its
//     much smaller error bound (node32_refine), and the populations the
//     decided alpha changes rewritten.
//   k_far_fixup: two lists of deferred nodes.  What the second stage left
//     open takes the FP64 series FORMULA (near64_formula), one node per
//     lane.  Nodes far from equilibrium (max |x_i| > 1/8, a velocity
//     component >= 1/4), invalid states and the rare node the series does
//     not settle take the FP64 FORMULA with logarithms, one node per warp.
//     alpha is rounded down to FP32.  It also resets the other parity's
//     counters for the next step (stream order makes them idle here).
#pragma once
#include <type_traits>
#include "sc32.cuh"
#include "series64.cuh"
#include "warp64.cuh"

namespace elbm {

// Second stage of one deferred node from its stored values v[] (FP32
// storage: the stored value; FP16: the decoded deviation); the kernel wrote
// it with the provisional alpha ap (NaN: unknown, recomputed).  Returns
// the second stage's status (kStageDone, kStageRetry: left to the FP64
// series, kStageFP64: left to the logarithms).
template <class L, bool SHIFTED, int DIAG, int CHECK, class A, class Out>
__device__ __forceinline__ int refine_deferred(const StepParams& p,
                                               const float (&v)[L::Q],
                                               long long node, float ap, A& acc,
                                               Out out) {
  auto in = [&](int i) { return v[i]; };
  return second_stage32<L, SHIFTED, DIAG, CHECK>(
      in, p.rho0f, p.betaf, p.corr_rho, p.corr,
      p.alpha_map ? p.alpha_map + node : nullptr, ap, out,
      [&](const N32<L>& r) {
        if (!DIAG) return;
        if constexpr (!std::is_same<A, Acc>::value) {
          diag32<L, SHIFTED, CHECK, true>(r, in, p.rho0, acc);
        } else {
          const double j[3] = {r.j[0], r.j[1], r.j[2]};
          acc.add_moments((double)r.drho, j, (double)r.rho);
          acc.add_alpha((double)r.alpha, r.flags, 0);
          if (CHECK) {
            Node64<L> nd;
            const Check64 ck = check32<L, SHIFTED>(in, p.rho0, r.alpha, nd);
            acc.add_check(ck.h, ck.violation,
                          decision_mismatch(r.flags, ck.accept_ref),
                          fabs((double)r.alpha - ck.alpha_ref));
          }
        }
      });
}

// Second stage of the undecided nodes in the buffer (S: the storage type,
// float or half_t).  Block b of the stream-collide launch (`blocks`
// blocks) wrote refine_counts[b] entries from b (refine_cap / blocks) on;
// every block of this kernel forms their prefix sums in shared memory and
// takes entries k with a grid stride.  The double-float stage decides (and
// rewrites the populations its alpha changes); the few nodes its FP32
// series leaves open join the open-node list (the queue's upper end), for
// the FP64 series in the fixup, whose register budget holds it.
template <class L, class S, int DIAG, int CHECK>
__global__ void __launch_bounds__(256, 2) k_refine_stage(const StepParams p,
                                                         int blocks) {
  chain_begin();
  constexpr int Q = L::Q;
  __shared__ unsigned pre[kMaxRefineBlocks + 1];
  block_prefix(p.refine_counts, blocks, pre);
  const unsigned total = pre[blocks];
  const unsigned seg = p.refine_cap / (unsigned)blocks;
  const bool shifted = sizeof(S) == 2 || !p.unshifted;
  Acc32T<Sum2> acc;
  acc.init();
  for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < total;
       k += gridDim.x * blockDim.x) {
    int lo = 0, hi = blocks;   // pre[lo] <= k < pre[lo + 1]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (pre[mid] <= k)
        lo = mid;
      else
        hi = mid;
    }
    constexpr int R = refine_record<L>();
    const float4* rec = reinterpret_cast<const float4*>(
        p.refine_buf + ((size_t)lo * seg + (k - pre[lo])) * (size_t)R);
    float w[R];
#pragma unroll
    for (int j = 0; j < R / 4; ++j) {
      const float4 t = rec[j];
      w[4 * j] = t.x;
      w[4 * j + 1] = t.y;
      w[4 * j + 2] = t.z;
      w[4 * j + 3] = t.w;
    }
    float v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = w[i];
    const long long node = __float_as_uint(w[Q]);
    const float ap = w[Q + 1];
    int st;
    if constexpr (sizeof(S) == 2) {
      st = refine_deferred<L, true, DIAG, CHECK>(
          p, v, node, ap, acc, [&](int i, float val) {
            reinterpret_cast<unsigned short*>(p.out_pop[i])[node] =
                h16_bits<L>(val, i);
          });
    } else {
      auto out = [&](int i, float val) { p.out_pop[i][node] = val; };
      st = shifted
               ? refine_deferred<L, true, DIAG, CHECK>(p, v, node, ap,
                                                              acc, out)
               : refine_deferred<L, false, DIAG, CHECK>(p, v, node, ap,
                                                               acc, out);
    }
    if (st != kStageDone) {
      // still open: list from the queue's top; far: list from its bottom
      const int open = st == kStageRetry;
      const unsigned q = atomicAdd(&p.far_count[2 * open + p.parity], 1u);
      if (q < p.far_cap)
        p.far_queue[open ? p.far_cap - 1u - q : q] = (unsigned)node;
      else
        atomicOr(p.err_flags, NF_BAD_NONFINITE);   // cannot happen: cap = n
    }
  }
  if (DIAG) store_acc32(acc, p.partials);
}

// FP64 fixup (S: the storage type, float or half_t); values are gathered
// from f_in.  The open-node list (what the second stage left) takes the FP64
// series, one node per lane.  Of the deferred-node queue, entries tagged
// kTagRefine (a full buffer segment, or no buffer) take the second stage
// here first, one per thread, and what it leaves is collected per warp for
// the series.  Nodes that need the logarithms are collided one at a time
// by their whole warp (formula64_warp, one population per lane), or one per
// lane when a warp has more than five, collected 32 at a time on a queue
// longer than the grid (the first step after initialisation).  On steps with
// the FP64 entropy check (CHECK) the logarithms run on their own lanes, so
// that the check repeats their very sums (a tie would otherwise count as a
// mismatch by rounding); the series forms are the other steps'.
//
// Bound by latency: a short list is one chain per warp, and by the fetch of
// straight-line code that each warp runs once.  A few open nodes run one
// at a time (near64_warp), many one per lane (near64_formula: up to 32 nodes
// for ~120 FP64 instructions of 64 cycles); the form is the list's, so the
// same input gives the same alphas.  (Logarithm nodes take the form their
// warp's share asks for: their sums, and a tie's branch, may differ by
// rounding between runs.)  Before, the second stage ran
// again with double-float leading terms (~3,000 FP32 instructions) and what
// that left took the logarithms, ~460 FP64 instructions a node.  Entries are
// dealt evenly as runs of neighbours; the grid is one block per SM (the
// kernel's registers allow no second one).
// us per launch, before -> now (GB300): D3Q27 256^3 binary16 41 -> 15,
// 121 x 64 x 70 static step (no buffer) 36 -> 22, D2Q9 1024^2 shear layer
// 25 -> 12; all open nodes one per lane: static 64.
// First step after initialisation (every node undecided, the logarithm nodes
// together in symmetry planes), before the FP64 series -> with partial flushes
// per warp -> runs dealt across blocks, remainders pooled, ties sent straight
// to the logarithms: Taylor-Green 96^3 445 -> 703 -> 380, 256^3
// 4000 -> 4590 -> 3700; random phases 96^3 184 -> 144 -> 155, 256^3
// 2340 -> 2020 -> 2100.
template <class L>
__device__ __forceinline__ void near64_gather(const StepParams& p, int x, int y,
                                              int z, const float*, double (&f)[L::Q]) {
#pragma unroll
  for (int i = 0; i < L::Q; ++i)
    f[i] = load64<L, float>(p.in_pop[i][src_index<L>(p, i, x, y, z)], i,
                            p.rho0, p.unshifted);
}
template <class L>
__device__ __forceinline__ void near64_gather(const StepParams& p, int x, int y,
                                              int z, const half_t*, double (&f)[L::Q]) {
#pragma unroll
  for (int i = 0; i < L::Q; ++i)
    f[i] = load64<L, half_t>(reinterpret_cast<const half_t*>(
                                 p.in_pop[i])[src_index<L>(p, i, x, y, z)],
                             i, p.rho0, false);
}

// FP64 entropy check (Eq. (7)) of a node at the alpha it took, from its stored
// values in f_in.
template <class L, class S>
__device__ __noinline__ Check64 check_stored(const StepParams& p,
                                             long long node, double alpha) {
  int x, y, z;
  node_xyz<L>(p, (unsigned)node, x, y, z);
  Node64<L> c;
  near64_gather<L>(p, x, y, z, static_cast<const S*>(nullptr), c.f);
  node64_prepare(c);
  return node64_check(c, alpha);
}

// Entries of a list of `count` that a warp of `warps` takes per round: runs
// of neighbouring entries, of equal length, at most 32.
__device__ __forceinline__ unsigned run_length(unsigned count, unsigned warps) {
  return min(32u, (count + warps - 1u) / warps);
}
// The run a warp takes.  Short lists: consecutive runs to different blocks, so
// that every SM has some (dealt block by block, steps of 189 x 107 x 83 and of
// the 12-member batch were 3 and 5 % longer).  Queues longer than the grid:
// four consecutive runs to a block, which share cache lines and run on its
// four sub-partitions (nodes that need the logarithms lie together, in a
// symmetry plane).
__device__ __forceinline__ unsigned dealt(bool bulk, unsigned warp) {
  return bulk ? ((warp >> 2) * gridDim.x + blockIdx.x) * 4u + (warp & 3u)
              : warp * gridDim.x + blockIdx.x;
}

// Open nodes per warp up to which they run one at a time (near64_warp) rather
// than one per lane (near64_formula).  us per step of 64,250 (D2Q9) and
// 65,600 (D3Q27) nodes with 1, 2, 5, 6 and 16 open nodes per warp, GB300:
//   D2Q9   in turn 27.1 34.4 57.3 63.9 136   per lane 28.1 28.9 30.1 29.3 29.9
//   D3Q27  in turn 36.3 41.7 57.4 66.7 114   per lane 51.8 55.1 58.3 61.0 71.1
template <class L>
__host__ __device__ constexpr unsigned few_open() {
  return L::Q == 9 ? 1u : 5u;
}
// The form is the whole list's, not a warp's: which entries share a warp is
// the order of atomic additions, and alphas of the two forms (~1e-15 apart)
// may round down to different FP32 numbers, so a choice per warp would let two
// runs of one input differ.
__device__ __forceinline__ bool few_listed(unsigned count, unsigned blocks,
                                           unsigned few) {
  return count <= blocks * (8u * few);
}
// Of `count` queued entries, which take the second stage here first, a few
// per cent are left open in a developed flow (under 2 per warp of two rounds);
// on a longer queue (the first step after initialisation) lanes fill up.
__device__ __forceinline__ bool few_queued(unsigned count, unsigned warps) {
  return count <= 64u * warps;
}
// Warps per block that take open nodes: all while each gets few, then one
// per sub-partition as long as their lanes hold the list (two would share
// the FP64 pipe for nothing), then all.
__device__ __forceinline__ unsigned open_warps(unsigned count, unsigned blocks,
                                               unsigned few) {
  return !few_listed(count, blocks, few) && count <= blocks * (4u * 32u) ? 4u
                                                                         : 8u;
}

template <class L, class S, int DIAG, int CHECK>
__global__ void __launch_bounds__(256) k_far_fixup(const StepParams p) {
  chain_begin();
  constexpr int Q = L::Q;
  const unsigned count = min(p.far_count[p.parity], p.far_cap);
  const unsigned open_count = min(p.far_count[2 + p.parity], p.far_cap);
  if (blockIdx.x == 0 && threadIdx.x < 2)
    p.far_count[2 * threadIdx.x + (p.parity ^ 1)] = 0u;
  if (count + open_count == 0u) {   // uniform: this row of statistics is empty
    if (DIAG && threadIdx.x < NSTAT)
      p.partials[(long long)blockIdx.x * NSTAT + threadIdx.x] =
          threadIdx.x == S_AMIN ? INFINITY
                                : (threadIdx.x == S_AMAX ? -INFINITY : 0.0);
    return;
  }
  const bool shifted = sizeof(S) == 2 || !p.unshifted;
  const int lane = threadIdx.x & 31;
  const unsigned W = gridDim.x * (blockDim.x >> 5);
  const LanePop lp = lane_pop<L>(lane);
  const bool bulk = count > gridDim.x * blockDim.x;
  Acc acc;
  acc.init();
  auto coords = [&](long long node, int& x, int& y, int& z) {
    node_xyz<L>(p, (unsigned)node, x, y, z);
  };
  auto out_s = [&](long long node, int i, float val) {
    if constexpr (sizeof(S) == 2)
      reinterpret_cast<unsigned short*>(p.out_pop[i])[node] =
          h16_bits<L>(val, i);
    else
      p.out_pop[i][node] = val;
  };
  // FP64 FORMULA of one node in this thread
  auto fp64_lane = [&](long long node) {
    int x, y, z;
    coords(node, x, y, z);
    Node64<L> nd;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const long long src = src_index<L>(p, i, x, y, z);
      double vi;
      if constexpr (sizeof(S) == 2)
        vi = h16_dev<L>(reinterpret_cast<const unsigned short*>(
                            p.in_pop[i])[src],
                        i);
      else
        vi = p.in_pop[i][src];
      nd.f[i] = shifted ? L::w(i) * p.rho0 + vi : vi;
    }
    auto store_s = [&](int i, double val) {
      if (i < 0) {
        p.alpha_map[node] = (float)val;
      } else if constexpr (sizeof(S) == 2) {
        reinterpret_cast<half_t*>(p.out_pop[i])[node] =
            h16_from_dev<L>(val - L::w(i) * p.rho0, i);
      } else {
        p.out_pop[i][node] =
            (float)(p.unshifted ? val : val - L::w(i) * p.rho0);
      }
    };
    if (DIAG) acc.far += 1;
    collide64<L, MODE_FORMULA, CHECK>(nd, p, true, acc, DIAG != 0, store_s);
  };
  auto check = [&](long long node, double alpha, unsigned flags) {
    const Check64 ck = check_stored<L, S>(p, node, alpha);
    acc.add_check(ck.h, ck.violation, decision_mismatch(flags, ck.accept_ref),
                  fabs(alpha - ck.alpha_ref));
  };
  // FP64 FORMULA of node nd by the whole warp (every lane calls): the series
  // form when `near` and it settles the node, else the logarithm form; with
  // CHECK the series form only.  Returns whether the node is done.
  auto fp64_warp = [&](long long nd, bool near, Warp64& r) {
    int x, y, z;
    coords(nd, x, y, z);
    double f = 0.0;
    if (lp.on) {
      int xs = x - lp.c[0], ys = y - lp.c[1], zs = z - lp.c[2];
      xs = xs < 0 ? xs + p.nx : (xs >= p.nx ? xs - p.nx : xs);
      ys = ys < 0 ? ys + p.ny : (ys >= p.ny ? ys - p.ny : ys);
      zs = zs < 0 ? zs + p.nz : (zs >= p.nz ? zs - p.nz : zs);
      const long long src = ((long long)zs * p.ny + ys) * p.nx + xs;
      if constexpr (sizeof(S) == 2) {
        const unsigned short b =
            reinterpret_cast<const unsigned short*>(p.in_pop[lane])[src];
        f = (double)(__half2float(__ushort_as_half(b)) * lp.hscale_inv);
      } else {
        f = (double)p.in_pop[lane][src];
      }
      if (shifted) f += lp.w * p.rho0;
    }
    auto store = [&](double val) {
      if constexpr (sizeof(S) == 2)
        reinterpret_cast<half_t*>(p.out_pop[lane])[nd] =
            __double2half((val - lp.w * p.rho0) * (double)lp.hscale);
      else
        p.out_pop[lane][nd] = (float)(p.unshifted ? val : val - lp.w * p.rho0);
    };
    const bool settled =
        near && near64_warp<L>(lp, lane, f, p.beta, r, store);
    if (CHECK && !settled) return false;
    if (!settled) r = formula64_warp<L>(lp, f, p.beta, store);
    if (lane == 0) {
      if (DIAG) acc.far += !settled;
      if (r.flags & (NF_BAD_NEG | NF_BAD_NONFINITE)) {
        atomicOr(p.err_flags, r.flags);
      } else {
        if (p.alpha_map) p.alpha_map[nd] = (float)r.alpha;
        if (DIAG) {
          acc.add_moments(r.rho - p.rho0, r.j, r.rho);
          acc.add_alpha(r.alpha, r.flags, 0);
        }
      }
    }
    return true;
  };
  // FP64 series FORMULA of one node in this thread; false: not settled
  auto near_lane = [&](long long node) {
    int x, y, z;
    coords(node, x, y, z);
    Near64<L> nd;
    near64_gather<L>(p, x, y, z, static_cast<const S*>(nullptr), nd.f);
    double alpha = 2.0;
    unsigned flags = NF_BAND;
    if (!near64_formula(nd, alpha, flags)) return false;
    const double ab = alpha * p.beta;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const double val = fma(ab, nd.n[i], nd.f[i]);
      if constexpr (sizeof(S) == 2)
        reinterpret_cast<half_t*>(p.out_pop[i])[node] =
            h16_from_dev<L>(fma(-L::w(i), p.rho0, val), i);
      else
        p.out_pop[i][node] =
            (float)(p.unshifted ? val : fma(-L::w(i), p.rho0, val));
    }
    if (p.alpha_map) p.alpha_map[node] = (float)alpha;
    if (DIAG) {
      const double j[3] = {nd.j[0] * nd.unit, nd.j[1] * nd.unit,
                           nd.j[2] * nd.unit};
      const double rho = nd.rho * nd.unit;
      acc.add_moments(rho - p.rho0, j, rho);
      acc.add_alpha(alpha, flags, 0);
      if (CHECK) check(node, alpha, flags);
    }
    return true;
  };
  // this warp's pending nodes (8 warps; warp-uniform counts): for the
  // logarithms (on a queue longer than the grid; at most 32 before a round
  // adds up to 32) and for the series (below 32 before)
  __shared__ unsigned pend_s[8][64], near_s[8][64];
  const int warp = threadIdx.x >> 5;
  unsigned* pend = pend_s[warp];
  unsigned* near = near_s[warp];
  int npend = 0, nnear = 0;
  auto flush = [&]() {   // 32 of them; every lane calls
    npend -= 32;
    __syncwarp();
    fp64_lane((long long)pend[npend + lane]);
    __syncwarp();
  };
  // Nodes that need the logarithms (every lane calls).  Per lane a node
  // costs ~75 FP64 warp instructions of its warp (2,400 shared by 32 lanes),
  // per warp ~460: one per warp ends sooner when a warp has few such nodes,
  // one per lane costs less FP64 issue in bulk.
  auto logarithms = [&](bool need64, long long node, bool near) {
    const unsigned m64 = __ballot_sync(0xffffffffu, need64);
    if (CHECK ? !near : (!bulk && !near && __popc(m64) > 5)) {
      if (need64) fp64_lane(node);
    } else if (bulk && !near) {
      const int nk = __popc(m64);
      if (npend + nk > 64) flush();
      if (need64) pend[npend + __popc(m64 & ((1u << lane) - 1u))] =
          (unsigned)node;
      npend += nk;
    } else {
      unsigned m = m64;
      double alpha = 2.0;      // with CHECK: what this lane's node took
      unsigned flags = 0u;
      while (m) {
        const int src_lane = __ffs(m) - 1;
        m &= m - 1;
        Warp64 r;
        const bool done =
            fp64_warp(__shfl_sync(0xffffffffu, node, src_lane), near, r);
        if (CHECK && done && lane == src_lane) {
          alpha = r.alpha;
          flags = r.flags;
          need64 = false;
        }
      }
      if (CHECK) {
        if (flags != 0u) check(node, alpha, flags);
        if (need64) fp64_lane(node);
      }
    }
  };
  // Rounds over the open-node list, then over the queue, then until the
  // nodes its second stage left are settled; one call site each for the
  // series and the logarithms.
  const unsigned use = open_warps(open_count, gridDim.x, few_open<L>());
  const bool few_o = few_listed(open_count, gridDim.x, few_open<L>());
  const bool few_q = few_queued(count, W);
  const unsigned WO = gridDim.x * use;
  const unsigned run_o = run_length(open_count, WO);
  const unsigned run_q = run_length(count, W);
  unsigned base_o = (unsigned)warp < use ? 0u : open_count, base_q = 0u;
  for (;;) {
    bool need64 = false, open = false, direct = false, few = few_o;
    long long node = 0;
    if (base_o < open_count) {
      const unsigned k =
          base_o + dealt(bulk, (unsigned)warp) * run_o + (unsigned)lane;
      base_o += run_o * WO;
      direct = (unsigned)lane < run_o && k < open_count;
      if (direct) node = p.far_queue[p.far_cap - 1u - k];
    } else if (base_q < count) {
      const unsigned k =
          base_q + dealt(bulk, (unsigned)warp) * run_q + (unsigned)lane;
      base_q += run_q * W;
      if ((unsigned)lane < run_q && k < count) {
        const unsigned e = p.far_queue[k];
        node = e & ~kTagRefine;
        need64 = true;
        if (e & kTagRefine) {
          int x, y, z;
          coords(node, x, y, z);
          float v[Q];
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            const long long src = src_index<L>(p, i, x, y, z);
            if constexpr (sizeof(S) == 2)
              v[i] = h16_dev<L>(reinterpret_cast<const unsigned short*>(
                                    p.in_pop[i])[src],
                                i);
            else
              v[i] = p.in_pop[i][src];
          }
          const float ap = __int_as_float(0x7fc00000);   // NaN: recomputed
          auto out = [&](int i, float val) { out_s(node, i, val); };
          const int st =
              shifted ? refine_deferred<L, true, DIAG, CHECK>(p, v, node, ap,
                                                              acc, out)
                      : refine_deferred<L, false, DIAG, CHECK>(p, v, node, ap,
                                                               acc, out);
          open = st == kStageRetry;
          need64 = st == kStageFP64;
        }
      }
    } else if (nnear == 0) {
      break;
    }
    // nodes for the series: this round's list entries, or a warp's worth
    // (at the end, the rest) of what the second stage left
    const unsigned mo = __ballot_sync(0xffffffffu, open);
    if (open)
      near[nnear + __popc(mo & ((1u << lane) - 1u))] = (unsigned)node;
    nnear += __popc(mo);
    long long sn = node;
    if (nnear >= 32 || (nnear > 0 && base_q >= count)) {   // warp-uniform
      const int take = min(nnear, 32);
      nnear -= take;
      few = few_q;
      __syncwarp();
      direct = lane < take;
      if (direct) sn = (long long)near[nnear + lane];
      __syncwarp();
    }
    if (!few) direct = direct && !near_lane(sn);
#pragma unroll 1
    for (int t = 0; t < 2; ++t)
      logarithms(t == 0 ? direct : need64, t == 0 ? sn : node, t == 0 && few);
  }
  // What the warps still hold of a long queue, pooled over the block: full
  // warps of nodes, one per lane, on different sub-partitions (few nodes: one
  // per warp).
  if (bulk) {
    __shared__ unsigned pool[8 * 64];
    __shared__ int held[8];
    if (lane == 0) held[warp] = npend;
    __syncthreads();
    int at = 0, total = 0;
    for (int w = 0; w < 8; ++w) {
      if (w < warp) at += held[w];
      total += held[w];
    }
    for (int k = lane; k < npend; k += 32) pool[at + k] = pend[k];
    __syncthreads();
    for (int k = 32 * warp; k < total; k += 32 * 8) {
      const int m = min(32, total - k);
      const unsigned e = lane < m ? pool[k + lane] : 0u;
      if (m > 5) {
        if (lane < m) fp64_lane((long long)e);
      } else {
        for (int j = 0; j < m; ++j) {
          Warp64 r;   // (with CHECK nothing is pending)
          fp64_warp((long long)__shfl_sync(0xffffffffu, e, j), false, r);
        }
      }
    }
  }
  if (DIAG) acc.block_reduce_store(p.partials);
}

}  // namespace elbm
