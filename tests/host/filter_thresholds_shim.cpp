// C entry points over csrc/filter_thresholds.h for the CPU tests (ctypes).
#include "filter_thresholds.h"

extern "C" {

// wrap_hi, wrap_lo and max_sq for a panorama width and a distance.
void ft_thresholds(int width, float max_px, float* out) {
    const pmsp::FilterThresholds t = pmsp::filter_thresholds(width, max_px);
    out[0] = t.wrap_hi;
    out[1] = t.wrap_lo;
    out[2] = t.max_sq;
}

}  // extern "C"
