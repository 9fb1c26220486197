// Docking-kernel instances for 16 lanes per start (9 to 16 torsion steps, two
// starts per warp): the group size is a constant.
#include "dock_kernel.cuh"

namespace ligate {

const void *dock_fn_l16(int mode, int minb) {
  switch (mode * 2 + (minb - 4)) {
    case 0: return (const void *)dock_kernel<MODE_F32_PLAIN, 4, 16>;
    case 1: return (const void *)dock_kernel<MODE_F32_PLAIN, 5, 16>;
    case 2: return (const void *)dock_kernel<MODE_F32_CORNER, 4, 16>;
    case 3: return (const void *)dock_kernel<MODE_F32_CORNER, 5, 16>;
    case 4: return (const void *)dock_kernel<MODE_BF16_CORNER, 4, 16>;
    case 5: return (const void *)dock_kernel<MODE_BF16_CORNER, 5, 16>;
    case 6: return (const void *)dock_kernel<MODE_F16_CORNER, 4, 16>;
    default: return (const void *)dock_kernel<MODE_F16_CORNER, 5, 16>;
  }
}

}  // namespace ligate
