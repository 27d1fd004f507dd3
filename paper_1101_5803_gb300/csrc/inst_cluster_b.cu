// cluster CGLS kernels, 5x5 and 19x19 PSFs
#include "cluster.cuh"
#include "table.h"

namespace mirage {
void fill_cluster_b(KernelTable& t) {
    t.cluster[5][0] = (const void*)k_cgls_cluster<5, 256>;
    t.cluster[5][1] = (const void*)k_cgls_cluster<5, 512>;
    t.cluster[19][0] = (const void*)k_cgls_cluster<19, 256>;
    t.cluster[19][1] = (const void*)k_cgls_cluster<19, 512>;
}
}  // namespace mirage
