// march_lattice_3d.cu -- instances of march_lattice_3d.cuh without a field per site.
#include "march_lattice_3d.cuh"

namespace ihmc {

int march3_lattice_threads(const Geometry &g) {
    if (g.dim != 3 || g.X % 4 != 0) return 0;
    const int T = m3_threads(g.X, g.Y);
    return T <= M3_THREADS && m3_smem(g.P, T) <= 227 * 1024 ? T : 0;
}

// Chains are split while that leaves at most one CTA per SM, or CTAs so small
// that their threads number below 352 per SM, each with four planes at least
// (four more than its own are computed per evaluation).  Trajectories of 64 chains,
// N_md = 10, at 1 / 2 / 4 CTAs per chain: L = 16 0.164 / 0.117 / 0.094 ms, 32
// 0.281 / 0.187 / 0.145, 48 0.746 / 0.457 / 0.542, 64 1.358 / 0.780 / 0.934.
int march3_lattice_split(const Geometry &g, int n_chains) {
    const int sms = sm_count();
    const int64_t T = m3_threads(g.X, g.Y);
    int cs = 1;
    while (cs < MAX_CS && g.nplanes >= 8 * cs &&
           (2 * cs * (int64_t)n_chains <= sms || 2 * cs * n_chains * T <= 352 * (int64_t)sms))
        cs *= 2;
    return cs;
}

cudaError_t march3_lattice_node(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    return a.hdf ? march3_node_field(a, np, args) : march3_node_plain(a, np, args);
}

cudaError_t march3_node_plain(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    const bool odd = a.g.Y % 2 != 0;
    if (a.cs > 1) return odd ? node3<true, false, true>(a, np, args) : node3<true, false, false>(a, np, args);
    return odd ? node3<false, false, true>(a, np, args) : node3<false, false, false>(a, np, args);
}

}  // namespace ihmc
