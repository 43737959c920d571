// march_lattice_3d.cu -- instances of march_lattice_3d.cuh without a field per site.
#include <algorithm>

#include "march_lattice_3d.cuh"

namespace ihmc {

int march3_lattice_threads(const Geometry &g) {
    if (g.dim != 3 || g.X % 4 != 0) return 0;
    const int T = m3_threads(g.X, g.Y);
    return T <= M3_THREADS && m3_smem(g.P, T) <= 227 * 1024 ? T : 0;
}

// CTAs resident on an SM: by threads (128 registers each) and shared memory.
static int march3_resident(const Geometry &g) {
    const int T = m3_threads(g.X, g.Y);
    return std::min(M3_THREADS / T, (int)(227 * 1024 / (m3_smem(g.P, T) + 1024)));
}

// Chains are split while that leaves at most one CTA per SM, or CTAs so small
// that their threads number at most 352 per SM, each with four planes at least
// (four more than its own are computed per evaluation), and all are resident at
// once, six at most on an SM.  Trajectories of 64 chains, N_md = 10, at 1 / 2 / 4 CTAs per
// chain: L = 16 0.164 / 0.117 / 0.094 ms, 32 0.281 / 0.187 / 0.145, 48 0.746 / 0.457 / 0.542, 64
// 1.358 / 0.780 / 0.934.  Against the plane-streaming kernel's time, nine evaluations: 200 chains of
// 32^3 (337 threads per SM once split) 0.70 / 0.54, of 28^3 0.80 / 0.63; 400 chains of 20^3 0.97 /
// 1.25 (five CTAs fit), of 16^3 0.92 / 0.80 / 1.12 (six); 304 chains of 8 x 8 x 20 0.96 / 0.69 /
// 1.03 (eight).
int march3_lattice_split(const Geometry &g, int n_chains) {
    const int64_t T = m3_threads(g.X, g.Y), sms = sm_count(), n = n_chains;
    const int64_t fit = sms * std::min(march3_resident(g), 6);
    int cs = 1;
    while (cs < MAX_CS && g.nplanes >= 8 * cs && 2 * cs * n <= fit &&
           (2 * cs * n <= sms || 2 * cs * n * T <= 352 * sms))
        cs *= 2;
    return cs;
}

// Planes of few tiles leave its CTAs with one or two warps and few of those fit on an
// SM, so many such chains, and a field's loads, which nothing hides, are the
// plane-streaming kernel's; where all CTAs are resident at once it holds its own.  Against
// that kernel's time, nine evaluations (with a field per site): 152 chains of 24^3 0.71 (0.89),
// 304 of 20^3 0.89 (1.00), of 24^3 0.91 (1.11), of 32^3 0.82 (0.98), 608 of 20^3 0.87 (1.10), of 16^3 0.94
// (1.13), 1000 of 16^3 (912 fit) 1.18 (1.54), of 12^3 0.90 (1.10), of 8 x 8 x 20 1.11 (1.30), of 28^3 0.82
// (1.05), of 32 x 32 x 16 0.65 (0.87); two evaluations, 304 of 24^3 1.11 (1.30).  Of fewer than
// eight planes the four extra ones of every evaluation eat the gain but for full, large
// planes (389 of 32 x 56 x 7 0.73).  With this rule 11 of 2402 lattices are slower by more than
// 3 % (the worst 1.25, with a sign flip per trajectory); 206 gains of 1662 are left out.
int march3_lattice_pays(const Geometry &g, int n_chains, int n_pass, bool field) {
    const int T = m3_threads(g.X, g.Y), tiles = (g.X / 4) * ((g.Y + 1) / 2);
    const int sms = sm_count(), per_sm = (n_chains + sms - 1) / sms, cs = march3_lattice_split(g, n_chains);
    const bool longer = n_pass >= 8, full = 8 * tiles >= 7 * T;
    if (g.nplanes < 8) return g.nplanes >= 6 && !field && T >= 128 && longer && full;
    if (T >= 256 || cs >= 4) return 1;
    if (field) {
        if (T >= 128) return (per_sm == 1 && (longer || T >= 192)) || (longer && full);
        return longer && cs >= 2 && per_sm <= 2 && (T >= 64 || g.nplanes >= 16);
    }
    if (T >= 128 || per_sm == 1) return 1;
    if (n_pass < 5) return 0;
    if (T >= 96) return longer || cs >= 2 || full;
    if (per_sm <= 2) return longer || cs >= 2;
    return longer && (per_sm <= 3 || (per_sm == 4 && g.nplanes >= 20) || (T == 64 && tiles == T) ||
                      (tiles >= 18 && n_chains <= sms * march3_resident(g)));
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
