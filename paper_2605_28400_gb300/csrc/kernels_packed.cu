// kernels_packed.cu — the packed int16x2 instantiations of the wavefront kernel (wavefront.cuh):
// two triplets per column task, one per 16-bit half, global alignment, score only. Compiled
// apart from the int32 instantiations.
#include "wavefront_vp.cuh"

namespace trioseq {

namespace {

template <int NJ, int NK>
const void* pptr(int mode) {
  if (mode == 2) return reinterpret_cast<const void*>(&wavefront_vp_kernel<NJ, NK>);
  if (mode == 1)
    return reinterpret_cast<const void*>(&wavefront_kernel<NJ, NK, false, kGlobal, 1, false>);
  return nullptr;
}

}  // namespace

const void* wavefront_packed(int nj, int nk, int mode) {
  if (nj == 8 && nk == 8) return pptr<8, 8>(mode);
  if (nj == 8 && nk == 4 && mode == 2) return pptr<8, 4>(2);
  if (nj == 4 && nk == 8) return pptr<4, 8>(mode);
  if (nj == 4 && nk == 4) return pptr<4, 4>(mode);
  return nullptr;
}

// sigma'' table, both triplets' 16-bit profiles, the staging ring, the residue ring
size_t wavefront_vp_smem_bytes(int nj, int nk, int KP) {
  const size_t sigN = (size_t)((KP * KP + 3) & ~3);
  const size_t prof = (size_t)KP * (kPR * (vp_repeat(KP) ? kPC : 1) * nj + kPC * nk);
  const size_t slot = (size_t)kPC * nk + kPC + (size_t)kPR * nj;
  return (sigN + prof + kRing * slot + 2 * kVpRing) * sizeof(int);
}

}  // namespace trioseq
