// cluster CGLS kernels, 3x3 and 21x21 PSFs
#include "cluster.cuh"
#include "table.h"

namespace mirage {
void fill_cluster_a(KernelTable& t) {
    t.cluster[3][0] = (const void*)k_cgls_cluster<3, 256>;
    t.cluster[3][1] = (const void*)k_cgls_cluster<3, 512>;
    t.cluster[21][0] = (const void*)k_cgls_cluster<21, 256>;
    t.cluster[21][1] = (const void*)k_cgls_cluster<21, 512>;
}
}  // namespace mirage
