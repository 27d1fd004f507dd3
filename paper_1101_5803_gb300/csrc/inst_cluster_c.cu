// cluster CGLS kernels, 7x7 and 17x17 PSFs
#include "cluster.cuh"
#include "table.h"

namespace mirage {
void fill_cluster_c(KernelTable& t) {
    t.cluster[7][0] = (const void*)k_cgls_cluster<7, 256>;
    t.cluster[7][1] = (const void*)k_cgls_cluster<7, 512>;
    t.cluster[17][0] = (const void*)k_cgls_cluster<17, 256>;
    t.cluster[17][1] = (const void*)k_cgls_cluster<17, 512>;
}
}  // namespace mirage
