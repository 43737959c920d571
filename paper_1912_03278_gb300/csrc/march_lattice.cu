// march_lattice.cu -- launch parameters of the 2D kernel that runs several force
// evaluations per sweep (march_lattice.cuh) and its instances for rows of whole
// vectors.
#include "march_lattice.cuh"

namespace ihmc {

// One thread per four columns, whole warps.
int march_lattice_threads(const Geometry &g) {
    if (g.dim != 2 || g.X > 4 * MARCH_CTA_THREADS || g.nplanes < 24) return 0;
    return ((g.X + 3) / 4 + 31) / 32 * 32;
}

cudaError_t march_lattice_node(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    const bool rag = a.g.X % 4 != 0;
    if (a.hdf) return rag ? march_node_rag_field(a, a.march, np, args) : march_node_vec_field(a, a.march, np, args);
    return rag ? march_node_rag(a, a.march, np, args) : march_node_vec(a, a.march, np, args);
}

cudaError_t march_node_vec(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args) {
    return node_ts<false, false>(a, T, np, args);
}

}  // namespace ihmc
