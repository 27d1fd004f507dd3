// The kernels of inst_fast.cu compiled for one CTA per SM:
//   fast[K][1][mode], for calls with no more items than SMs
#include "fast.cuh"
#include "table.h"

namespace mirage {
void fill_fast1(KernelTable& t) {
    t.fast[5][1][0] = (const void*)k_cgls_fast<5, 4, TAPS_SMEM_X2, 1>;
    t.fast[7][1][0] = (const void*)k_cgls_fast<7, 4, TAPS_SMEM_X2, 1>;
    t.fast[9][1][0] = (const void*)k_cgls_fast<9, 4, TAPS_SMEM_X2, 1>;
    t.fast[11][1][0] = (const void*)k_cgls_fast<11, 4, TAPS_SMEM_X2, 1>;
    t.fast[9][1][1] = (const void*)k_cgls_fast<9, 4, TAPS_PARAM, 1>;
    t.fast[9][1][2] = (const void*)k_cgls_fast<9, 4, TAPS_PARAM_X2, 1>;
    t.fast[9][1][3] = (const void*)k_cgls_fast<9, 4, TAPS_PARAM_TF32, 1>;
    t.fast[5][1][2] = (const void*)k_cgls_fast<5, 4, TAPS_PARAM_X2, 1>;
    t.fast[7][1][2] = (const void*)k_cgls_fast<7, 4, TAPS_PARAM_X2, 1>;
    t.fast[11][1][2] = (const void*)k_cgls_fast<11, 4, TAPS_PARAM_X2, 1>;
}
}  // namespace mirage
