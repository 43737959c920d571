// march_lattice_3d_field.cu -- instances of march_lattice_3d.cuh with a field per site.
#include "march_lattice_3d.cuh"

namespace ihmc {

cudaError_t march3_node_field(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    const bool odd = a.g.Y % 2 != 0;
    if (a.cs > 1) return odd ? node3<true, true, true>(a, np, args) : node3<true, true, false>(a, np, args);
    return odd ? node3<false, true, true>(a, np, args) : node3<false, true, false>(a, np, args);
}

}  // namespace ihmc
