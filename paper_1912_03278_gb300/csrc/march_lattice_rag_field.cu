// march_lattice_rag_field.cu -- instances of march_lattice.cuh: ragged rows, a field per site.
#include "march_lattice.cuh"

namespace ihmc {

cudaError_t march_node_rag_field(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args) {
    return node_ts<true, true>(a, T, np, args);
}

}  // namespace ihmc
