// kernels_vl.cu — global score instantiations of the two-cells-per-register kernel
// (wavefront_vl.cuh): 8 rows x 2 x 8 columns per lane (column tasks of 32 x 128 cells), 8 rows x
// 2 x 4 (32 x 64), 4 rows x 2 x 4 (16 x 64), and the 32 x 128 tasks with the lane's sigma''(y,z) tile
// and row-major profiles in shared memory (2-warp CTAs, 5 per SM, or 1-warp CTAs, 9 per SM).
// Traceback keys and the other alignment types compile apart (kernels_vl_tb.cu, kernels_vl_types.cu).
#include "wavefront_vl.cuh"

namespace trioseq {

namespace {
template <int NJ, int NH, int CS>
const void* vptr() {
  return reinterpret_cast<const void*>(&wavefront_vl_kernel<NJ, NH, CS, kGlobal, false>);
}
}  // namespace

// cs: sigma''(y,z) tile in shared memory, 2-warp CTAs (1, tile label "8x16s") or 1-warp CTAs
// (2, "8x16t"); 0: in registers
const void* wavefront_vl(int nj, int nk, int cs, int at, bool tb) {
  if (tb) return at == kGlobal && cs == 0 ? wavefront_vl_tb(nj, nk) : nullptr;
  if (at != kGlobal) return cs == 0 ? wavefront_vl_types(nj, nk, at) : nullptr;
  if (nj == 8 && nk == 16) {
    if (cs == 1) return vptr<8, 8, 1>();
    if (cs == 2) return vptr<8, 8, 2>();
    return vptr<8, 8, 0>();
  }
  if (nj == 8 && nk == 8 && cs == 0) return vptr<8, 4, 0>();
  if (nj == 4 && nk == 8 && cs == 0) return vptr<4, 4, 0>();
  return nullptr;
}

int wavefront_vl_warps(int cs) {
  return cs == 1 ? VlLaunch<8, 8, 1>::warps : VlLaunch<8, 8, 0>::warps;
}

namespace {
template <int NJ, int NH, int CS>
size_t vl_smem(int KP) {
  using G = VlGeom<NJ, NH>;
  const size_t sigN = (size_t)((KP * KP + 3) & ~3);
  const size_t prof = !CS ? (size_t)KP * (kPR * kPC * NJ / 2 + kPC * NH)
                          : (size_t)KP * (G::PJ16 + G::PK16) / 2;
  const size_t cv = CS ? (size_t)32 * 4 * G::CVG : 0;
  return (sigN + (size_t)VlLaunch<NJ, NH, CS>::warps * (prof + kRing * G::SLOT + kVlRing + cv)) * sizeof(int);
}
}  // namespace

size_t wavefront_vl_smem_bytes(int nj, int nk, int KP, int cs) {
  if (nj == 8 && nk == 16)
    return cs == 1 ? vl_smem<8, 8, 1>(KP) : (cs == 2 ? vl_smem<8, 8, 2>(KP) : vl_smem<8, 8, 0>(KP));
  if (nj == 8 && nk == 8 && cs == 0) return vl_smem<8, 4, 0>(KP);
  if (nj == 4 && nk == 8 && cs == 0) return vl_smem<4, 4, 0>(KP);
  return 0;
}

}  // namespace trioseq
