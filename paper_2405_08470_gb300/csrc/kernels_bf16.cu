// kernels_bf16.cu - BF16-factor instantiations of the fused spMTTKRP + remap
// kernels (factor rows stored in BF16, products and sums in FP32).
#include "mttkrp_direct.cuh"
#include "mttkrp_kernel.cuh"

namespace spm {

static int launch_direct_bfloat16(const MttkrpArgs& a, const LaneCfg& c, cudaStream_t s) {
  if (c.vec) {
    switch (a.nmodes) {
      case 3:
        if (a.es == 16) return launch_direct<3, __nv_bfloat16, 8, 1, 4>(a, c.L, s);
        return launch_direct<0, __nv_bfloat16, 8, 1, 2>(a, c.L, s);
      case 4: return launch_direct<4, __nv_bfloat16, 8, 1, 4>(a, c.L, s);
      case 5: return launch_direct<5, __nv_bfloat16, 8, 1, 4>(a, c.L, s);
      case 6: return launch_direct<6, __nv_bfloat16, 8, 1, 4>(a, c.L, s);
      default: return launch_direct<0, __nv_bfloat16, 8, 1, 2>(a, c.L, s);
    }
  }
  switch (c.RC) {
    case 1: return launch_direct<0, __nv_bfloat16, 1, 1, 2>(a, c.L, s);
    case 2: return launch_direct<0, __nv_bfloat16, 1, 2, 2>(a, c.L, s);
    case 4: return launch_direct<0, __nv_bfloat16, 1, 4, 2>(a, c.L, s);
    default: return launch_direct<0, __nv_bfloat16, 1, 8, 2>(a, c.L, s);
  }
}

int launch_mttkrp_bf16(const MttkrpArgs& a, const LaneCfg& c, cudaStream_t s) {
  if (a.loss_part) {  // fused CP-loss pass (3 modes, 16- or 32-byte nonzeros, vector lanes)
    if (!(c.vec && a.nmodes == 3 && (a.es == 32 || a.es == 16)))
      return fail(SPM_ERR_UNSUPPORTED,
                  "fused CP-loss pass: 3 modes, 16- or 32-byte nonzeros only");
    if (a.es == 16) {
      if (c.VW == 4) {
        switch (a.mode) {
          case 0: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 0, 16, true>(a, c.L, s);
          case 1: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 1, 16, true>(a, c.L, s);
          default: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 2, 16, true>(a, c.L, s);
        }
      }
      switch (a.mode) {
        case 0: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 0, 16, true>(a, c.L, s);
        case 1: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 1, 16, true>(a, c.L, s);
        default: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 2, 16, true>(a, c.L, s);
      }
    }
    if (c.VW == 4) {
      switch (a.mode) {
        case 0: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 0, 32, true>(a, c.L, s);
        case 1: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 1, 32, true>(a, c.L, s);
        default: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 2, 32, true>(a, c.L, s);
      }
    }
    switch (a.mode) {
      case 0: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 0, 32, true>(a, c.L, s);
      case 1: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 1, 32, true>(a, c.L, s);
      default: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 2, 32, true>(a, c.L, s);
    }
  }
  if (a.variant == 3) {  // form 3: one remap warp per CTA (the dispatcher checked the layout)
    if (c.VW == 4) {
      switch (a.mode) {
        case 0: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 0, 32, false, true>(a, c.L, s);
        case 1: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 1, 32, false, true>(a, c.L, s);
        default:
          return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 2, 32, false, true>(a, c.L, s);
      }
    }
    switch (a.mode) {
      case 0: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 0, 32, false, true>(a, c.L, s);
      case 1: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 1, 32, false, true>(a, c.L, s);
      default: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 2, 32, false, true>(a, c.L, s);
    }
  }
  if (a.variant == 1) return launch_direct_bfloat16(a, c, s);
  if (c.VW < 4 && narrow_built(a, c)) return launch_narrow_bf16(a, c, s);
  if (c.vec && c.VW == 4) {  // 8-byte lane slices: the FP32 kernel's lane shape
    switch (a.nmodes) {
      case 3:
        if (warp_steps(a, c) == 4) {  // one-lane groups
          switch (a.mode + (a.es == 32 ? 0 : 3)) {
            case 0: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 0, 32>(a, c.L, s);
            case 1: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 1, 32>(a, c.L, s);
            case 2: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 2, 32>(a, c.L, s);
            case 3: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 0, 16>(a, c.L, s);
            case 4: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 1, 16>(a, c.L, s);
            default: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 4, 2, 16>(a, c.L, s);
          }
        }
        if (a.es == 32) {
          switch (a.mode) {
            case 0: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 0, 32>(a, c.L, s);
            case 1: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 1, 32>(a, c.L, s);
            default: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 2, 32>(a, c.L, s);
          }
        }
        switch (a.mode) {
          case 0: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 0, 16>(a, c.L, s);
          case 1: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 1, 16>(a, c.L, s);
          default: return launch_warp_kernel<3, __nv_bfloat16, 4, 1, 8, 2, 16>(a, c.L, s);
        }
      case 4: return launch_modes<4, __nv_bfloat16, 4, 4>(a, c.L, s);
      case 5: return launch_modes<5, __nv_bfloat16, 4, 4>(a, c.L, s);
      case 6: return launch_modes<6, __nv_bfloat16, 4, 4>(a, c.L, s);
      default: return launch_any_modes<__nv_bfloat16, 4>(a, c, s);
    }
  }
  if (c.vec && c.VW == 8) {
    switch (a.nmodes) {
      case 3:
        // 4 steps of 16 bytes: with 8 the scratch holds 2 of them and its loop stands four
        // times in the kernel (10M nonzeros at R 64: 1.31 ms per sweep, 0.90 with 4)
        if (a.es == 32) {  // elements padded to a full 32-byte sector
          switch (a.mode) {
            case 0: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 0, 32>(a, c.L, s);
            case 1: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 1, 32>(a, c.L, s);
            default: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 2, 32>(a, c.L, s);
          }
        }
        switch (a.mode) {
          case 0: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 0, 16>(a, c.L, s);
          case 1: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 1, 16>(a, c.L, s);
          default: return launch_warp_kernel<3, __nv_bfloat16, 8, 1, 4, 2, 16>(a, c.L, s);
        }
      case 4: return launch_modes<4, __nv_bfloat16, 8, 4>(a, c.L, s);
      case 5: return launch_modes<5, __nv_bfloat16, 8, 4>(a, c.L, s);
      case 6: return launch_modes<6, __nv_bfloat16, 8, 2>(a, c.L, s);
      default: return launch_warp_kernel<0, __nv_bfloat16, 8, 1, 4>(a, c.L, s);
    }
  }
  if (c.vec) return launch_any_modes<__nv_bfloat16, 2>(a, c, s);
  switch (c.RC) {
    case 1: return launch_any_modes<__nv_bfloat16, 1>(a, c, s);
    case 2: return launch_warp_kernel<0, __nv_bfloat16, 1, 2, 4>(a, c.L, s);
    case 4: return launch_warp_kernel<0, __nv_bfloat16, 1, 4, 4>(a, c.L, s);
    default: return launch_warp_kernel<0, __nv_bfloat16, 1, 8, 2>(a, c.L, s);
  }
}

}  // namespace spm
