// FP64 panel solve, 8 right-hand sides a CTA (see panel_kernel.cuh; one file per few widths, compiled in
// parallel).
#include "panel_kernel.cuh"

namespace gb {
template int launch_panel_cw<double, 8>(const Canon<double> &, int64_t, int, double);
}  // namespace gb
