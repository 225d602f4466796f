// The solver's on-chip form with a label cost (nu > 0), in a translation unit of
// its own so that its instantiations compile beside the others'.
#include "seg_tile.cuh"

SegPlan seg_plan_mdl(int H, int W, int n, int n_sm) { return seg_plan_t<true>(H, W, n, n_sm); }
