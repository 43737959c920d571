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

// Rows of whole vectors: always, but for short trajectories in a field per site of many
// chains (1000 chains, two evaluations: 256 x 40 1.20 of the plane-streaming kernel's time,
// 128 x 64 1.05; without a field 0.9).  Ragged rows fill a quarter of the lanes
// that the plane-streaming kernel (a site per lane) fills, draw two random
// blocks where it draws one, and the instances spill, so they pay where the chain is cut
// into slabs (which takes 48 rows, and chains few enough) or sweeps of three evaluations
// outweigh the dearer first and last ones.  This kernel / plane-streaming, nine
// evaluations: 152 chains of 31 x 96 0.36 (with a field 0.54), 99 x 64 0.61 (0.81), 99 x 24 1.16
// (1.45), 255 x 24 0.92 (1.17), 301 x 24 0.68 (0.85); 608 of 61 x 64 0.87 (1.03), 1000 of 31 x 64
// 1.41 (1.73), of 61 x 64 1.04 (1.30), of 99 x 64 0.61 (0.80), of 255 x 28 0.50 (0.76); two
// evaluations, 1000 of 61 x 60 1.82 (1.88), 21: 1000 of 61 x 60 0.79 (1.08).  With this rule one of
// 5961 is slower by more than 3 % (by 3.5); 548 gains of 3802 are left out.
int march_lattice_pays(const Geometry &g, int n_chains, int n_pass, bool field) {
    const int sms = sm_count(), per_sm = (n_chains + sms - 1) / sms;
    if (g.X % 4 == 0) return !(field && n_pass <= 4 && per_sm >= 5);
    const int warps = (g.X + 31) / 32, rows = g.nplanes;   // warps of a row in the other kernel
    const bool cut = rows >= 2 * MARCH_MIN_SLAB, tall = rows >= 4 * MARCH_MIN_SLAB, longer = n_pass >= 9;
    if (warps > 8) return cut || !field || n_pass >= 5 || per_sm > 2;
    if (warps > 4) {
        if (cut) return !field || longer || (tall && (per_sm <= 2 || n_pass >= 5));
        if (per_sm >= (field ? 8 : 4)) return 1;
        return field ? longer && per_sm >= (n_pass >= 20 ? 2 : 4) : n_pass >= 6;
    }
    if (cut && per_sm <= 2) return !field || longer || tall;
    if (warps > 2) {
        if (cut) return field ? longer : n_pass >= 5;
        return (longer && per_sm >= (field ? 5 : 2)) || (n_pass >= 20 && !field);
    }
    if (!cut) return warps == 2 && !field && n_pass >= 18;
    if (per_sm == 3) return longer || (tall && n_pass >= 5);
    if (warps == 2)
        return field ? n_pass >= 20 && (per_sm <= 4 || per_sm >= 14)
                     : n_pass >= 15 || (longer && per_sm == 4) || (tall && n_pass >= 6 && per_sm >= 8);
    const bool few = 2 * (int64_t)n_chains <= 7 * (int64_t)sms;   // (still cut into five slabs)
    return field ? tall && few && n_pass >= 20 : n_pass >= 30 || (tall && few && longer);
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
