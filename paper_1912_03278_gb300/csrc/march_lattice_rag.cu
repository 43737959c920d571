// march_lattice_rag.cu -- instances of march_lattice.cuh: ragged rows.
#include "march_lattice.cuh"

namespace ihmc {

cudaError_t march_node_rag(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args) {
    return node_ts<true, false>(a, T, np, args);
}

}  // namespace ihmc
