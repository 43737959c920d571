// tiny_lattice.cu -- FP32 HMC trajectories on small lattices, the whole chain on
// chip: psi and u in shared memory, every thread's own psi and p in registers.
//
// The streaming kernels walk through a chain plane by plane, which on a lattice
// of 16 x 16 is 20 dependent steps of almost no work per force evaluation (0.8 us
// each).  Here all sites are updated at once, two barriers per evaluation; HBM is
// touched once per trajectory (the proposal and the end momenta, which stay
// readable).  64 chains of 16 x 16, N_md = 5, eight trajectories: 0.09 ms, on the
// plane-streaming kernel 0.71.  Latency bounds it: two warps on each of 64 SMs, issue 14 % of
// the cycles, stalls per issue wait 2.9, barrier 1.2, short scoreboard 1.0, no instruction
// 0.9; 117 registers, no spills.
//
// psi and p are computed by its operations in the same order and agree bit for
// bit.  So do the estimators' compensated FP32 sums: Kahan's scheme rounds every
// addend, so the per-vector terms are left in shared memory and summed in the
// order of the plane-streaming kernel's threads.
#include "march_lattice.cuh"

namespace ihmc {
namespace {

constexpr int TINY_THREADS = 512;

// V sites per item (consecutive, of one row): 4 where rows split into vectors.
template <int V>
struct Item {
    float x[V], p[V];
};

struct TinySmem {
    float *psi, *u, *est;   // est: vT, vAT, vHT of every item
};

// Neighbour sum of the item's sites in the order of gather() (fused_lattice_impl.cuh).
template <int DIM, int V>
__device__ __forceinline__ void tiny_gather(const Geometry &g, const float *f, int i0, int e0, Nbr<DIM, V> &n) {
    const int P = g.P, N = (int)g.N;
    const float *pc = f + (i0 - e0);   // e0: offset in the plane
    const float *pm = i0 - e0 == 0 ? f + (N - P) : pc - P;
    const float *pq = i0 - e0 + P == N ? f : pc + P;
    gather<DIM, V>(g, pm, pc, pq, e0, DIM == 2 ? e0 : e0 % g.X, n);
}

template <int DIM, int V, int QPT>
__global__ void __launch_bounds__(TINY_THREADS)
    tiny_kernel(const __grid_constant__ FusedArgs A, const __grid_constant__ Schedule S) {
    extern __shared__ float4 smem_f4[];
    const Geometry &g = A.g;
    const int T = blockDim.x, tid = threadIdx.x, N = (int)g.N, items = N / V;
    for (int i = tid; i < LOG1PEXP_NODES; i += T) smem_f4[i] = A.lpe_tab[i];
    const float4 *tab = smem_f4;
    TinySmem sm;
    sm.psi = reinterpret_cast<float *>(smem_f4 + LOG1PEXP_NODES);
    sm.u = sm.psi + (N + 3) / 4 * 4;
    sm.est = sm.u + (N + 3) / 4 * 4;
    double *red = reinterpret_cast<double *>(sm.est + (3 * items + 3) / 4 * 4);
    int *bcast = reinterpret_cast<int *>(red + 32 * 8);
    const int chain = A.chain0 + (int)blockIdx.x;
    if (chain >= A.n_chains) return;
    ChainState *const st = A.state + chain;
    const ChainParams prm = A.params[chain];
    const ActConst kc = act_const(prm);
    const double invN = 1.0 / (double)N;
    const int64_t cbase = (int64_t)chain * g.N;
    const bool has_h = A.hdf || !kc.hzero;

    Item<V> it[QPT];
    int e0[QPT];
#pragma unroll
    for (int k = 0; k < QPT; ++k) e0[k] = (tid + k * T) * V % g.P;
    // own items into registers and shared memory
    auto load = [&](int buf) {
        const float *src = sel3(A, buf) + cbase;
#pragma unroll
        for (int k = 0; k < QPT; ++k) {
            const int v = tid + k * T;
            if (v >= items) break;
            const Vec<V> t = ldv<V>(src + v * V);
#pragma unroll
            for (int q = 0; q < V; ++q) it[k].x[q] = t.v[q];
            stv<V>(sm.psi + v * V, t);
        }
    };
    auto field = [&](int i) { return A.hdf ? prm.betaf * A.hdf[i].x : prm.hpf; };
    // This thread's share of the action of sign * psi (in shared memory) and of the
    // estimators' sums.
    auto action = [&](float sign, uint32_t traj, uint64_t seed, double (&w)[5]) {
        Acc acc = acc_zero();
#pragma unroll 1
        for (int k = 0; k < QPT; ++k) {
            const int v = tid + k * T;
            if (v >= items) break;
            Nbr<DIM, V> n;
            tiny_gather<DIM, V>(g, sm.psi, v * V, v * V % g.P, n);
            Acc one = acc_zero();   // its estimator sums: the item's terms alone
            one.S = acc.S;
            one.Slo = acc.Slo;
            one.sS = acc.sS;
            vector_action<DIM, V>(A, kc, n, v * V, sign, traj, seed, chain, tab, one);
            acc.S = one.S;
            acc.Slo = one.Slo;
            acc.sS = one.sS;
            sm.est[v] = one.sT;   // (first addend of a compensated sum: exact)
            sm.est[items + v] = one.sAT;
            sm.est[2 * items + v] = one.sHT;
        }
        __syncthreads();
        // the plane-streaming kernel's thread t owned items t, t + nt, ... of
        // every plane
        const int nvec = g.P / V, nt = min(256, (nvec + 31) / 32 * 32);
        float s[3] = {0.0f, 0.0f, 0.0f}, c[3] = {0.0f, 0.0f, 0.0f};
        if (tid < nt && tid < nvec)
            for (int z = 0; z < g.nplanes; ++z)
                for (int e = tid; e < nvec; e += nt)
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        if (j < 2 || has_h) kahan_add(s[j], c[j], sm.est[j * items + z * nvec + e]);
        w[0] = acc_val(acc.S, acc.Slo);
        for (int j = 0; j < 3; ++j) w[1 + j] = kahan_val(s[j], c[j]);
        w[4] = (double)acc.sS;
    };

    int start = st->start;
    double S_cur = st->S;
    load(start);
    __syncthreads();
    if (A.eval_start) {
        double ev[5];
        action(1.0f, TRAJ_INIT, 0, ev);
        block_sum<5>(ev, red);
        S_cur = ev[0];
        if (tid == 0) {
            st->S = ev[0];
            set_obs(st, prm, ev[1], ev[2], ev[3], ev[4], invN);
            st->prop = start;
        }
    }
    for (int j = 0; j < A.n_traj; ++j) {
        const uint32_t traj = A.traj0 + (uint32_t)j;
        // ---- momenta (Sec. 3) ----
        f2 K{0.0f, 0.0f};
        float Klo = 0.0f;
#pragma unroll 1
        for (int k = 0; k < QPT; ++k) {
            const int v = tid + k * T;
            if (v >= items) break;
            const Vec<V> z = draw_momenta<V>(v * V, traj, chain, A.seed);
            stv<V>(sm.u + v * V, z);   // through u: the draw's code appears once
        }
#pragma unroll
        for (int k = 0; k < QPT; ++k) {
            const int v = tid + k * T;
            if (v >= items) break;
            const Vec<V> z = ldv<V>(sm.u + v * V);
#pragma unroll
            for (int q = 0; q < V; ++q) {
                it[k].p[q] = z.v[q];
                acc_add(K, Klo, two_prod(z.v[q], 0.5f * z.v[q]));
            }
        }
        const double K0 = acc_val(K, Klo);
        // ---- force evaluations ----
        for (int s = 0; s < S.n_pass; ++s) {
            const float kick = (float)(S.kick[s] * prm.eps), drift = (float)(S.drift[s] * prm.eps);
#pragma unroll
            for (int k = 0; k < QPT; ++k) {
                const int v = tid + k * T;
                if (v >= items) break;
                Nbr<DIM, V> n;
                tiny_gather<DIM, V>(g, sm.psi, v * V, e0[k], n);
                Vec<V> u;
#pragma unroll
                for (int q = 0; q < V; ++q)
                    u.v[q] = tanh_f(fmaf(prm.Cf, n.c.v[q], fmaf(prm.bJf, n.nb.v[q], field(v * V + q)))) - n.c.v[q];
                stv<V>(sm.u + v * V, u);
            }
            __syncthreads();
            const bool last = s + 1 == S.n_pass;
#pragma unroll
            for (int k = 0; k < QPT; ++k) {
                const int v = tid + k * T;
                if (v >= items) break;
                Nbr<DIM, V> n;
                tiny_gather<DIM, V>(g, sm.u, v * V, e0[k], n);
                Vec<V> x;
#pragma unroll
                for (int q = 0; q < V; ++q) {
                    const float F = fmaf(prm.Cf, n.c.v[q], prm.bJf * n.nb.v[q]);
                    it[k].p[q] = fmaf(kick, F, it[k].p[q]);
                    if (!last) it[k].x[q] = fmaf(drift, it[k].p[q], it[k].x[q]);
                    x.v[q] = it[k].x[q];
                }
                if (!last) stv<V>(sm.psi + v * V, x);
            }
            __syncthreads();
        }
        // ---- proposal out, energies, decision ----
        const int prop = buf_loc(start, S.n_pass - 1);
        float *gx = sel3(A, prop) + cbase, *gp = A.p + cbase;
        K = f2{0.0f, 0.0f};
        Klo = 0.0f;
#pragma unroll
        for (int k = 0; k < QPT; ++k) {
            const int v = tid + k * T;
            if (v >= items) break;
            Vec<V> x, p;
#pragma unroll
            for (int q = 0; q < V; ++q) {
                x.v[q] = it[k].x[q];
                p.v[q] = it[k].p[q];
                acc_add(K, Klo, two_prod(p.v[q], 0.5f * p.v[q]));
            }
            stv<V>(gx + v * V, x);
            stv<V>(gp + v * V, p);
        }
        double w[5];
        action(1.0f, traj, A.seed, w);
        double v7[7] = {K0, acc_val(K, Klo), w[0], w[1], w[2], w[3], w[4]};
        block_sum<7>(v7, red);
        const int cur = metropolis_step(CtaThreads{}, A, st, prm, chain, traj, start, prop, v7, invN, S_cur, true,
                                        bcast);
        if (cur == start) load(start);   // rejected
        start = cur;
        __syncthreads();
        if (A.flip_every > 0 && ((traj + 1) % (uint32_t)A.flip_every) == 0) {
            double wf[5];
            action(-1.0f, traj, A.seed, wf);
            block_sum<5>(wf, red);
            if (flip_step(CtaThreads{}, A, st, prm, chain, traj, wf, invN, S_cur, true, bcast)) {
                const int f = (start != prop) ? 3 - start - prop : (start + 1) % 3;
                float *gf = sel3(A, f) + cbase;
#pragma unroll
                for (int k = 0; k < QPT; ++k) {
                    const int v = tid + k * T;
                    if (v >= items) break;
                    Vec<V> x;
#pragma unroll
                    for (int q = 0; q < V; ++q) x.v[q] = it[k].x[q] = -it[k].x[q];
                    stv<V>(gf + v * V, x);
                    stv<V>(sm.psi + v * V, x);
                }
                start = f;
                if (tid == 0) st->start = f;
            }
            __syncthreads();
        }
        measure_step(CtaThreads{}, A, st, traj, true);
    }
}

template <int DIM, int V, int QPT>
cudaError_t tiny_node(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args) {
    auto kern = tiny_kernel<DIM, V, QPT>;
    static DeviceOnce once;
    const cudaError_t e = allow_smem(once, kern, 227 * 1024);
    if (e != cudaSuccess) return e;
    const int N = (int)a.g.N, items = N / V;
    np->func = reinterpret_cast<void *>(kern);
    np->gridDim = dim3((unsigned)(a.n_chains - a.chain0), 1, 1);
    np->blockDim = dim3((unsigned)T, 1, 1);
    np->sharedMemBytes = (unsigned)(LOG1PEXP_NODES * 16 + 2 * ((N + 3) / 4 * 4) * 4 +
                                    (3 * items + 3) / 4 * 4 * 4 + RED_BYTES);
    np->kernelParams = args;
    np->extra = nullptr;
    return cudaSuccess;
}

template <int DIM, int V>
cudaError_t tiny_qpt(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    const int items = (int)a.g.N / V;
    int T = (items + 31) / 32 * 32;
    if (T <= TINY_THREADS) return tiny_node<DIM, V, 1>(a, T, np, args);
    T = ((items + 1) / 2 + 31) / 32 * 32;
    if (T <= TINY_THREADS) return tiny_node<DIM, V, 2>(a, T, np, args);
    return tiny_node<DIM, V, 4>(a, TINY_THREADS, np, args);
}

}  // namespace

// Where it is the faster one.  It costs about 20 us per trajectory plus the work of
// the SM's chains (a site's action is its dearest part); the plane-streaming kernel the
// latency of a plane per evaluation, 0.4 us, and of the energies, so it gains with
// few planes, few evaluations and several chains per SM.  Measured over 5204 lattices,
// chains, fields and lengths of trajectory, this kernel / plane-streaming: one chain
// per SM 0.1 .. 0.9, but 600 x 3 with two evaluations 1.25, 1024 x 8 1.09; two chains
// per SM 64 x 64, nine evaluations 0.28, 16^3 0.87, but 16 x 16 x 8 1.16, 512 x 16 with two
// evaluations 1.50.  Many chains: only short rows or planes, which leave the
// lanes of the other kernel idle (4096 of 16 x 16, nine evaluations 0.25; 1000 of 32 x 64 0.67, with
// two evaluations 1.29; 1000 of 16 x 8 x 8 1.40; 3000 of 15 x 17 1.05).  With this rule none of
// them is slower by more than 3 %; 234 gains of 4656 are left out.
int tiny_lattice_fits(const Geometry &g, int n_chains, int n_pass) {
    const bool v4 = g.X % 4 == 0 && g.P % 4 == 0;
    if ((g.dim != 2 && g.dim != 3) || g.N > (int64_t)TINY_THREADS * 4 * (v4 ? 4 : 1)) return 0;
    const int sms = sm_count(), per_sm = (n_chains + sms - 1) / sms;
    const int nvec = g.P / (v4 ? 4 : 1);   // lanes that a plane fills in the other kernel
    const int64_t planes = (int64_t)g.nplanes * n_pass;
    const bool small = g.N <= (v4 ? 1024 : 256);
    if (per_sm <= 2 && small) return 1;
    if (per_sm == 1) return planes >= 24;
    if (per_sm == 2) return 3 * planes >= 5 * nvec + 12;
    if (!small && !(v4 && g.dim == 2 && g.X <= 32)) return 0;
    if (nvec <= 5 || (nvec <= 16 && n_pass >= 6 && (v4 || per_sm <= 8))) return 1;
    return nvec <= 36 && n_pass >= 9 && per_sm <= 3;
}

cudaError_t tiny_lattice_node(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    const bool v4 = a.g.X % 4 == 0 && a.g.P % 4 == 0;
    if (a.g.dim == 3) return v4 ? tiny_qpt<3, 4>(a, np, args) : tiny_qpt<3, 1>(a, np, args);
    return v4 ? tiny_qpt<2, 4>(a, np, args) : tiny_qpt<2, 1>(a, np, args);
}

}  // namespace ihmc
