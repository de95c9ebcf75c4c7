// Order 0 with one window of up to 4 x 4 cells (lpa_mean.cuh).
#include "lpa_mean.cuh"

const void *lpa_mean_wide(const LpaLaunch &L) { return lpa::pick<4, 3, false>(L); }
