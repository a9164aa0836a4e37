// Kernels of the mixed solver's dataflow iterations with register rows
// (cgp_flow.cuh): one kernel for each number of rows a thread may hold, so that
// each has the register file to itself (one kernel with all of them spills).
#include "cgp_flow.cuh"

namespace cgp {
namespace {

template <int R>
__global__ void __launch_bounds__(MAX_BLOCK) mixed_flow_kernel(Desc d) {
  __shared__ Shared sh;
  mark_pending(d, blockIdx.x);
  solve_mixed_flow<1, R>(d, blockIdx.x, sh);
}

// Many systems in one launch, as pcg_batched_kernel.
template <int R>
__global__ void __launch_bounds__(MAX_BLOCK)
    mixed_flow_batched_kernel(const Desc* __restrict__ descs, const int* __restrict__ blk_inst,
                              unsigned long long* t_start) {
  __shared__ Shared sh;
  if (t_start && blockIdx.x == 0 && threadIdx.x == 0) *t_start = global_ns();
  const Desc& d = descs[blk_inst[blockIdx.x]];
  const int lb = blockIdx.x - d.blk0;
  mark_pending(d, lb);
  solve_mixed_flow<1, R>(d, lb, sh);
}

template <int R>
const void* pick(bool batched) {
  return batched ? (const void*)mixed_flow_batched_kernel<R> : (const void*)mixed_flow_kernel<R>;
}

}  // namespace

// Kernel for blocks of `block` threads with at most `chunk` rows, one lane per
// row; NULL where a thread would hold more rows than are worth registers.  At
// 866 rows a block (two a thread) register rows take an iteration from 2.84 to
// 2.55 us; with four rows a thread the spills cost more than the shared-memory
// reads they save (8.3k against 7.4k clocks at 1732 rows a block).
const void* mixed_flow_kernel_ptr(int chunk, int block, bool batched) {
  if (block < kFlowMinBlock) return nullptr;
  const int per = (chunk + block - 1) / block;
  if (per <= 1) return pick<1>(batched);
  if (per <= 2) return pick<2>(batched);
  return nullptr;
}

}  // namespace cgp
