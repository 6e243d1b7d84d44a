// jx_batch_kernels.cu — the batched kernels (env groups of different sizes in one
// launch: steps by blocks of a few envs, the rest persistent over per-group
// work queues) and their launches.
#include "jx_device.cuh"

namespace jx {
namespace {

// One reset, render or rollout launch over the groups of a batch. Each group has a work queue (a
// counter of handed-out envs); a warp drains the groups' queues in order,
// one env at a time, fetching its next ticket while it works on the current
// env. The last warp to finish zeroes the counters for the next launch.
// SPEC 0: each group's map kind and grayscale stack as its Params say; SPEC 1:
// every group has bit-plane maps and no grayscale stack (compiled in).
template <int MODE, int COLS, int SPEC>
__global__ void __launch_bounds__(kBatchMaxThreads, kBatchMinBlocks)
    batch_kernel(const __grid_constant__ BatchParams bp) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  uint8_t* const wbase = smem_raw + warp * bp.warp_bytes;
  init_warp_header(wbase, lane);
  if (MODE == MODE_ROLLOUT) {  // after the walk and the draw: only the envs they left
    uint32_t left = 0u;
    for (int g = 0; g < bp.n_groups; ++g) {
      const Params& p = bp.g[g];
      if (p.stop == nullptr)
        left = 1u;
      else
        for (int i = lane; i < (p.n + 31) >> 5; i += 32) left |= p.ended[i];
    }
    if (!__any_sync(0xffffffffu, left != 0u)) return;  // the whole grid
  }
  const int gw = blockIdx.x * wpb + warp;
  int slot = 0;
  bool fresh = true;  // nothing of an earlier group is pending in the ring
  bool lost = false;  // a map copy of this warp was lost: it takes no further env
  for (int g = 0; g < bp.n_groups && !lost; ++g) {
    const Params& p = bp.g[g];
    uint32_t ticket = 0;
    if (lane == 0) {
      // a drained queue is skipped without an atomic
      ticket = *reinterpret_cast<volatile uint32_t*>(bp.queue + g);
      if (ticket < (uint32_t)p.n) ticket = atomicAdd(bp.queue + g, 1u);
    }
    ticket = __shfl_sync(0xffffffffu, ticket, 0);
    if (ticket >= (uint32_t)p.n) continue;
    if (!fresh && lane == 0) bulk_wait_read_all();  // the layout changes under the ring
    __syncwarp();
    write_palette(p, WarpSmem{wbase, fill_lane(p, lane)}, lane);
    fresh = false;
    slot = 0;
    uint8_t* scratch = p.gen_scratch ? p.gen_scratch + (size_t)gw * p.gen_scratch_stride : nullptr;
    while (ticket < (uint32_t)p.n) {
      uint32_t next = 0;
      if (lane == 0) next = atomicAdd(bp.queue + g, 1u);
      const int e = (int)ticket;
      const int first = MODE == MODE_ROLLOUT && p.stop != nullptr ? p.stop[e] : 0;
      if (MODE == MODE_ROLLOUT && first >= p.steps)
        ;  // all of its steps are drawn
      else if (SPEC == 1)
        lost = !run_env<MODE, MAP_BITS, COLS, 0>(p, e, wbase, scratch, lane, slot, first, p.steps);
      else
        lost = !run_env<MODE, MAP_RUNTIME, COLS, 2>(p, e, wbase, scratch, lane, slot, first, p.steps);
      if (lost) break;  // the counters are still cleared below: every warp reaches the end
      ticket = __shfl_sync(0xffffffffu, next, 0);
    }
  }
  if (lane == 0) {
    bulk_wait_read_all();
    __threadfence();
    const uint32_t nw = gridDim.x * wpb;
    if (atomicAdd(bp.queue + kMaxGroups, 1u) == nw - 1) {
      for (int g = 0; g < bp.n_groups; ++g) atomicExch(bp.queue + g, 0u);
      atomicExch(bp.queue + kMaxGroups, 0u);
    }
  }
}

// One step of every env of a batch: a warp an env, the blocks of the groups one
// after another, handed out as slots free: 74 us a step of 16 groups of 1024
// envs, 138 through the queues above, which serialise on their counters (every
// warp tries every group's). A warp's group, known from the block index, is
// uniform, so its parameters are read without indexing. A step is a
// programmatic dependent like the env kernel's.
template <int COLS, int SPEC>
__global__ void __launch_bounds__(kBatchMaxThreads, kBatchMinBlocks)
    batch_step_kernel(const __grid_constant__ BatchParams bp) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int g = 0;
  while (g + 1 < bp.n_groups && (int)blockIdx.x >= bp.first_block[g + 1]) ++g;
  const Params& p = bp.g[g];
  uint8_t* const wbase = smem_raw + warp * bp.warp_bytes;
  write_palette(p, WarpSmem{wbase, FillLane{}}, lane);
  if (SPEC == 0 && !p.map_bits && p.S * p.S >= 4096) init_warp_header(wbase, lane);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int e = ((int)blockIdx.x - bp.first_block[g]) * (int)(blockDim.x >> 5) + warp;
  if (e >= p.n) return;
  int slot = 0;
  if (SPEC == 1)
    run_env<MODE_STEP, MAP_BITS, COLS, 0>(p, e, wbase, nullptr, lane, slot);
  else
    run_env<MODE_STEP, MAP_RUNTIME, COLS, 2>(p, e, wbase, nullptr, lane, slot);
  if (lane == 0) bulk_wait_read_all();
}

auto batch_step_kernel_of(int cols, int spec) {
  if (spec == 1) return cols == 2 ? batch_step_kernel<2, 1> : batch_step_kernel<1, 1>;
  return cols == 2 ? batch_step_kernel<2, 0> : batch_step_kernel<1, 0>;
}

template <int MODE>
auto batch_kernel_for(int cols, int spec) {
  if (spec == 1) return cols == 2 ? batch_kernel<MODE, 2, 1> : batch_kernel<MODE, 1, 1>;
  return cols == 2 ? batch_kernel<MODE, 2, 0> : batch_kernel<MODE, 1, 0>;
}

auto batch_kernel_of(int mode, int cols, int spec) {
  switch (mode) {
    case MODE_RESET: return batch_kernel_for<MODE_RESET>(cols, spec);
    case MODE_ROLLOUT: return batch_kernel_for<MODE_ROLLOUT>(cols, spec);
    case MODE_RENDER: return batch_kernel_for<MODE_RENDER>(cols, spec);
    default: return batch_step_kernel_of(cols, spec);
  }
}
}  // namespace

int batch_spec(const BatchParams& bp) {
  for (int g = 0; g < bp.n_groups; ++g)
    if (!bp.g[g].map_bits || bp.g[g].gray) return 0;
  return 1;
}

cudaError_t batch_blocks_per_sm(int mode, int cols, int spec, int warps, int smem_bytes, int* blocks) {
  auto k = batch_kernel_of(mode, cols, spec);
  cudaError_t err = raise_smem_limit(k);
  if (err != cudaSuccess) return err;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k, 32 * warps, smem_bytes);
}

cudaError_t batch_step_launch(BatchParams& bp, int cols, int warps, cudaStream_t stream) {
  int64_t blocks = 0;
  for (int g = 0; g < bp.n_groups; ++g) {
    bp.first_block[g] = (int32_t)blocks;
    blocks += (bp.g[g].n + warps - 1) / warps;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)(32 * warps));
  cfg.dynamicSmemBytes = (size_t)bp.warp_bytes * warps;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, batch_step_kernel_of(cols, batch_spec(bp)), bp);
}

cudaError_t batch_launch(const BatchParams& bp, int mode, int cols, int warps, int grid, cudaStream_t stream) {
  batch_kernel_of(mode, cols, batch_spec(bp))<<<grid, 32 * warps, (size_t)bp.warp_bytes * warps, stream>>>(bp);
  return cudaGetLastError();
}
}  // namespace jx
