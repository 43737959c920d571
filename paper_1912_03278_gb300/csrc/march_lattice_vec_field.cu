// march_lattice_vec_field.cu -- instances of march_lattice.cuh: rows of whole vectors, a field per site.
#include "march_lattice.cuh"

namespace ihmc {

cudaError_t march_node_vec_field(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args) {
    return node_ts<false, true>(a, T, np, args);
}

}  // namespace ihmc
