// cluster CGLS kernels, 11x11 and 13x13 PSFs
#include "cluster.cuh"
#include "table.h"

namespace mirage {
void fill_cluster_e(KernelTable& t) {
    t.cluster[11][0] = (const void*)k_cgls_cluster<11, 256>;
    t.cluster[11][1] = (const void*)k_cgls_cluster<11, 512>;
    t.cluster[13][0] = (const void*)k_cgls_cluster<13, 256>;
    t.cluster[13][1] = (const void*)k_cgls_cluster<13, 512>;
}
}  // namespace mirage
