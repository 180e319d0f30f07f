// The binary64 transport kernel with virtual packets (a translation unit of its
// own, compiled beside the other).
#include "mc_transport_kernel.cuh"

namespace mcgpu {

const void *select_virtual_kernel(int line_mode, bool jb, bool rec) {
  if (line_mode == 0) return select_lines<0, true>(jb, rec);
  return line_mode == 2 ? select_lines<2, true>(jb, rec) : select_lines<1, true>(jb, rec);
}

}  // namespace mcgpu
