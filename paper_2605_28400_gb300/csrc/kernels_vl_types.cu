// kernels_vl_types.cu — the two-cells-per-register kernel (wavefront_vl.cuh) for the semi-global and
// local types, score only.
#include "wavefront_vl.cuh"

namespace trioseq {

namespace {
template <int AT>
const void* pick_tile(int nj, int nk) {
  if (nj == 8 && nk == 16)
    return reinterpret_cast<const void*>(&wavefront_vl_kernel<8, 8, 0, AT, false>);
  if (nj == 8 && nk == 8)
    return reinterpret_cast<const void*>(&wavefront_vl_kernel<8, 4, 0, AT, false>);
  if (nj == 4 && nk == 8)
    return reinterpret_cast<const void*>(&wavefront_vl_kernel<4, 4, 0, AT, false>);
  return nullptr;
}
}  // namespace

const void* wavefront_vl_types(int nj, int nk, int at) {
  if (at == kSemiGlobal) return pick_tile<kSemiGlobal>(nj, nk);
  if (at == kLocal) return pick_tile<kLocal>(nj, nk);
  return nullptr;
}

}  // namespace trioseq
