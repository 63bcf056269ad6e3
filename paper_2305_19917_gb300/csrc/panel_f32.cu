// FP32 panel solve (see panel_kernel.cuh).
#include "panel_kernel.cuh"

namespace gb {
template int launch_panel_cw<float, 4>(const Canon<float> &, int64_t, int, float);
template int launch_panel_cw<float, 8>(const Canon<float> &, int64_t, int, float);
}  // namespace gb
