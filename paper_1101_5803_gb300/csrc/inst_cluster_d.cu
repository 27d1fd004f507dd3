// cluster CGLS kernels, 9x9 and 15x15 PSFs
#include "cluster.cuh"
#include "table.h"

namespace mirage {
void fill_cluster_d(KernelTable& t) {
    t.cluster[9][0] = (const void*)k_cgls_cluster<9, 256>;
    t.cluster[9][1] = (const void*)k_cgls_cluster<9, 512>;
    t.cluster[15][0] = (const void*)k_cgls_cluster<15, 256>;
    t.cluster[15][1] = (const void*)k_cgls_cluster<15, 512>;
}
}  // namespace mirage
