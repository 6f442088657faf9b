// kernels_vl_tb.cu — the two-cells-per-register kernel with traceback keys (wavefront_vl.cuh): 8 or 4
// rows x 2 x 4 columns per lane, global type.
#include "wavefront_vl.cuh"

namespace trioseq {

const void* wavefront_vl_tb(int nj, int nk) {
  if (nj == 8 && nk == 8)
    return reinterpret_cast<const void*>(&wavefront_vl_kernel<8, 4, 0, kGlobal, true>);
  if (nj == 4 && nk == 8)
    return reinterpret_cast<const void*>(&wavefront_vl_kernel<4, 4, 0, kGlobal, true>);
  return nullptr;
}

}  // namespace trioseq
