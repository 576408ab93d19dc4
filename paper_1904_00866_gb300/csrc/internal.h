// Internal declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>

#include <string>

#include "stream_collide.cuh"

namespace elbm {

// Launch counter shared by all launch sites.
void count_launch();
void count_launches(long long n);

// Launch of a kernel that begins with chain_begin() (stats.cuh).  `chained`:
// the operation before it in the stream is another kernel of the same call,
// and its blocks may be scheduled while that kernel's last ones run
// (programmatic dependent launch); they wait there until it has completed
// and its writes are visible, so only the launch latency overlaps.  us per
// step (GB300), without -> with it, three flows: D2Q9 64^2 FP64 (two kernels)
// 12.3 -> 9.7; D3Q27 32^3 FP32 (four) 38-40 -> 35.5; D3Q27 96^3 108 -> 103;
// D2Q9 1024^2 shear layer 67-68 -> 64.
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), int grid, int block,
                                  size_t smem, cudaStream_t s, int chained,
                                  const A&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute a = {};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = chained ? 1 : 0;
  count_launch();
  const cudaError_t e = cudaLaunchKernelEx(&c, kernel, args...);
  const cudaError_t last = cudaGetLastError();
  return e != cudaSuccess ? e : last;
}

// Message returned by elbm_last_error(NULL) (thread-local).
void set_global_error(const std::string& msg);

// Whether the kernels of a step over `bytes` of populations are chained: up
// to 128 MB.  Small steps gain the launch latency (D2Q9 64^2: 21 %; D3Q27 32^3,
// 3.5 MB: 6-11 %; 96^3, 96 MB: 5 %); beyond, it is below 3 % of the step, and the next
// kernel's waiting blocks cost more than that (D3Q27 189 x 107 x 83, 181 MB:
// 2.88 ms per 20 steps without, 2.97 with; the batch's steps 4.64 and 5.25,
// so its launches are never chained).
inline int chain_pays(double bytes) { return bytes <= 128e6; }

// Sum `rows` partial rows (NSTAT doubles each) into out[NSTAT].
cudaError_t launch_finish(const double* partials, int rows, double* out,
                          int chained, cudaStream_t s);

// Public statistics record from the NSTAT reduced slots.
void stats_from_slots(const double* slots, double rho0, long long n,
                      long long step, int checked, void* out_stats);

// Per-translation-unit launchers.  grid <= 0 picks the occupancy-sized grid
// (SM count x resident blocks, capped by the work); *grid_used receives it.
#define ELBM_DECLARE_LAUNCHERS(LAT)                                          \
  cudaError_t launch_fp32_formula_##LAT(int diag, int check,                 \
                                        const StepParams& p, int grid,        \
                                        int block, cudaStream_t s,            \
                                        int* grid_used);                      \
  cudaError_t launch_far_##LAT(int diag, int check, const StepParams& p,     \
                               int grid, cudaStream_t s);                    \
  cudaError_t launch_fp32_fp64mode_##LAT(int mode, int diag, int check,      \
                                         const StepParams& p, int grid,       \
                                         int block, cudaStream_t s,           \
                                         int* grid_used);                     \
  cudaError_t launch_fp64_##LAT(int mode, int diag, int check,               \
                                const StepParams& p, int grid, int block,     \
                                cudaStream_t s, int* grid_used);              \
  cudaError_t launch_fp16_formula_##LAT(int diag, int check,                 \
                                        const StepParams& p, int grid,        \
                                        cudaStream_t s, int* grid_used);      \
  cudaError_t launch_far16_##LAT(int diag, int check, const StepParams& p,   \
                                 int grid, cudaStream_t s);                  \
  cudaError_t launch_fp16_fp64mode_##LAT(int mode, int diag, int check,      \
                                         const StepParams& p, int grid,       \
                                         int block, cudaStream_t s,           \
                                         int* grid_used);
ELBM_DECLARE_LAUNCHERS(d2q9)
ELBM_DECLARE_LAUNCHERS(d3q27)
#undef ELBM_DECLARE_LAUNCHERS

// Second stage of the undecided nodes a step buffered (D3Q27 and large
// binary16 D2Q9 lattices; the other D2Q9 kernels run it themselves).
cudaError_t launch_refine_d3q27(int diag, int check, const StepParams& p,
                                int blocks, int grid, cudaStream_t s);
cudaError_t launch_refine16_d2q9(int diag, int check, const StepParams& p,
                                 int blocks, int grid, cudaStream_t s);
cudaError_t launch_refine16_d3q27(int diag, int check, const StepParams& p,
                                  int blocks, int grid, cudaStream_t s);

cudaError_t launch_fp64_d1q3(int mode, int diag, int check,
                             const StepParams& p, int grid, int block,
                             cudaStream_t s, int* grid_used);

}  // namespace elbm
