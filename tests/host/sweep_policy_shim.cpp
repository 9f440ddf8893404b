// C entry points over csrc/sweep_policy.h for the CPU tests (ctypes).
#include "sweep_policy.h"

extern "C" {

int sw_bounded_serves(int views, int side, long long tiles, int sms) { return pmsp::bounded_serves(views, side, tiles, sms); }
long long sw_bounded_from(int w, int h) { return pmsp::bounded_from(w, h); }
float sw_close_cost() { return pmsp::CLOSE_COST; }

}  // extern "C"
