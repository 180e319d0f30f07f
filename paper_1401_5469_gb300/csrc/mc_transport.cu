// The binary64 transport kernel without virtual packets, and the launches of
// both precisions.
#include "mc_transport_kernel.cuh"

namespace mcgpu {

namespace {

// tables: the model's branching tables (bucket slots) are there
const void *select_kernel(int line_mode, int precision, bool jb, bool rec, bool tables, bool virt, int L) {
  if (precision == 1) return select_mixed_kernel(line_mode, jb, rec, L);
  if (virt) return select_virtual_kernel(line_mode, jb, rec);
  if (line_mode == 0) return select_lines<0, false>(jb, rec);
  if (line_mode == 2) return select_lines<2, false>(jb, rec);
  if (tables) return select_lines<1, false>(jb, rec);
  return jb ? kernel_ptr<3, true, false, false>() : kernel_ptr<3, false, false, false>();  // (no packet records)
}

size_t smem_bytes(int S, int precision, bool virt) {
  // binary64: shell tables, then per warp a lone walk's state and draws, and the
  // queued launches of v-packets
  return precision == 1 ? mixed_smem_bytes(S)
                        : shell_words(S) * sizeof(double) +
                              (kBlock / 32) * (kLoneBytes + (virt ? kVirtualQueue * sizeof(VirtualLaunch) : 0));
}

}  // namespace

int transport_block_size() { return kBlock; }

cudaError_t transport_occupancy(int line_mode, int precision, bool j_blue, bool record, bool tables, int S, int L,
                                int *blocks_per_sm) {
  const void *k = select_kernel(line_mode, precision, j_blue, record, tables, false, L);
  const size_t smem = smem_bytes(S, precision, false);
  if (smem > 48 * 1024) {  // the query, like the launch, needs the opt-in above 48 KB
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, kBlock, smem);
}

cudaError_t launch_transport(const TransportParams &p, int line_mode, int precision, bool j_blue,
                             bool record, int grid, int block, cudaStream_t st) {
  // the shared-memory layout (one draw buffer per warp) is sized for kBlock
  if (block != kBlock) return cudaErrorInvalidValue;
  const bool virt = p.n_virtual > 0;
  const void *k = select_kernel(line_mode, precision, j_blue, record, p.dbr_rec != nullptr, virt, p.L);
  const size_t smem = smem_bytes(p.S, precision, virt);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  void *args[] = {const_cast<TransportParams *>(&p)};
  return cudaLaunchKernel(k, dim3(grid), dim3(block), args, smem, st);
}

}  // namespace mcgpu
