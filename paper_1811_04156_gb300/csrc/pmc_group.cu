// Instances of the group chain kernel (pmc_group.cuh): 8 lanes per chain, the
// general physics.
#include "pmc_group.cuh"

namespace pmc {
namespace PMC_VARIANT {

size_t group_smem_bytes(bool grad, int smem_cap, int warps_per_block) {
  return static_cast<size_t>(warps_per_block) * (32 / kGroupLanes) *
         group_words(chain_arrays(true, grad), smem_cap) * sizeof(float);
}

cudaError_t group_kernel(bool grad, bool spill, const ChainParams* p, int grid, int warps_per_block, int smem_cap,
                         int* blocks_per_sm, cudaStream_t s) {
  const size_t smem = group_smem_bytes(grad, smem_cap, warps_per_block);
  if (spill)
    return grad ? group_call<true, true>(p, grid, warps_per_block, smem, blocks_per_sm, s)
                : group_call<false, true>(p, grid, warps_per_block, smem, blocks_per_sm, s);
  return grad ? group_call<true, false>(p, grid, warps_per_block, smem, blocks_per_sm, s)
              : group_call<false, false>(p, grid, warps_per_block, smem, blocks_per_sm, s);
}

}  // namespace PMC_VARIANT
}  // namespace pmc
