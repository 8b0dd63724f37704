// kernels_narrow_f32.cu - the warp-block kernel with lanes of one or two FP32 values per
// load: ranks that are no multiple of four, or factors aligned to less than 16 bytes.
// The modes are compile-time constants and the gathers of a whole chunk are in flight,
// as on the wide lanes; the runtime-modes kernel, which serves the other shapes, gathers
// mode after mode.  Measured in FP32: 3M nonzeros of 10007 x 30011 x 1009 at rank 25,
// 1.49 ms per sweep there and 0.41 here; 5M of 50021 x 4001 x 20011 at rank 50, one mode
// without remap, 0.93 and 0.22.
#include "mttkrp_kernel.cuh"

namespace spm {

template <int VW, int RC, int U>
static int launch_steps(const MttkrpArgs& a, int L, cudaStream_t s) {
  switch (a.nmodes) {
    case 3: return launch_warp_kernel<3, float, VW, RC, U>(a, L, s);
    case 4: return launch_warp_kernel<4, float, VW, RC, U>(a, L, s);
    case 5: return launch_warp_kernel<5, float, VW, RC, VW * RC == 1 ? U : 4>(a, L, s);
    default: return launch_warp_kernel<6, float, VW, RC, VW * RC == 1 ? U : 4>(a, L, s);
  }
}

template <int VW, int RC>
static int launch_narrow(const MttkrpArgs& a, const LaneCfg& c, cudaStream_t s) {
  if constexpr (RC == 1)  // (only a one-piece row can have one-lane groups)
    if (c.L == 1) return launch_steps<VW, RC, 4>(a, c.L, s);
  return launch_steps<VW, RC, 8>(a, c.L, s);
}

int launch_narrow_f32(const MttkrpArgs& a, const LaneCfg& c, cudaStream_t s) {
  if (c.VW == 2) return launch_narrow<2, 1>(a, c, s);
  return c.RC == 1 ? launch_narrow<1, 1>(a, c, s) : launch_narrow<1, 2>(a, c, s);
}

}  // namespace spm
