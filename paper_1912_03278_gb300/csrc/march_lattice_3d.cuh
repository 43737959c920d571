// march_lattice_3d.cuh -- FP32 HMC trajectories on 3D lattices whose rows are a
// multiple of four long, marching through the planes with register windows.
//
// A thread owns a 4 x 2 tile of every plane (four consecutive sites of two
// neighbouring rows) and marches along z: the neighbours along z and between
// the tile's rows are its own registers.  The rows before and after the tile
// come from shared memory -- psi from the planes as they were copied in, u from
// two alternating planes that the threads write -- and the ends of the tile's
// rows from edge values that the neighbouring threads publish (march_lattice.cuh).
// Per plane and eight sites that is 12 shared loads and 6 stores; the
// plane-streaming kernel (fused_lattice_impl.cuh) loads every neighbour.  One
// barrier per plane.  A chain can be split over a cluster of CTAs, a slab of
// planes each, as there.
//
// psi and p are computed by the operations of the plane-streaming kernel in
// the same order and agree bit for bit.
//
// What bounds it: HBM where the planes of all chains do not stay in L2 (152 chains of
// 64^3: 6.5 TB/s in the middle evaluations); else the latency of one plane after
// the other at four to sixteen warps per SM (64 chains of 32^3 on four CTAs each: 147 us per
// trajectory of 11 evaluations, issue 33 %, DRAM 1 %, stalls wait 1.3, long
// scoreboard 0.6, barrier 0.5 per issue).  128 registers; spills 336 .. 452 bytes a
// thread (stores; loads 344 .. 616), with a field 512 .. 604 (528 .. 728), in the first and
// last evaluations' draws and action.
#pragma once
#include "march_lattice.cuh"

namespace ihmc {
namespace {

constexpr int M3_THREADS = 512;   // at most: 128 registers a thread
constexpr int M3_RING = 4;        // planes of psi and of p in shared memory

// Threads of a CTA: one per tile, whole warps.
__host__ __device__ constexpr int m3_threads(int X, int Y) { return ((X / 4) * ((Y + 1) / 2) + 31) / 32 * 32; }
// Shared memory (bytes): table, psi and p planes, two u planes, edge values
// [2][row][end][thread], reduction words.
__host__ __device__ constexpr size_t m3_smem(int P, int T) {
    return (size_t)LOG1PEXP_NODES * 16 + (size_t)(2 * M3_RING + 2) * P * 4 + (size_t)T * 8 * 8 + RED_BYTES;
}

struct Tile {
    int tid, e[2];        // plane offsets of the tile's rows
    int ym, yp;           // of the rows before and after the tile
    int left, right;      // neighbouring threads
    int rows;             // rows of the tile that exist (0: idle thread)
};
__device__ __forceinline__ Tile make_tile(const Geometry &g) {
    const int nx = g.X / 4, ny = (g.Y + 1) / 2;
    const int t = threadIdx.x;
    const bool live = t < nx * ny;
    const int ty = live ? t / nx : 0, tx = live ? t - ty * nx : 0;
    Tile c;
    c.tid = t;
    c.rows = live ? (2 * ty + 1 < g.Y ? 2 : 1) : 0;
    c.e[0] = 2 * ty * g.X + 4 * tx;
    c.e[1] = c.rows == 2 ? c.e[0] + g.X : c.e[0];
    c.ym = ty == 0 ? c.e[0] + g.P - g.X : c.e[0] - g.X;
    c.yp = c.e[1] + g.X >= g.P ? c.e[1] + g.X - g.P : c.e[1] + g.X;
    c.left = live ? (tx == 0 ? t + nx - 1 : t - 1) : t;
    c.right = live ? (tx == nx - 1 ? t - (nx - 1) : t + 1) : t;
    return c;
}

__device__ __forceinline__ Row row_add(const Row &a, const Row &b) { return Row{add2(a.a, b.a), add2(a.b, b.b)}; }

struct March3Args {
    const float *src;      // psi read (chain base)
    float *dst, *p;        // psi written, momenta (chain base)
    uint32_t traj;
    float *ring, *ring_p, *u;   // psi planes, p planes, u planes
    float2 *edge;
    int z0, nz;            // the slab's planes
};

// One force evaluation over the slab's planes (roles of FIRST, LAST, EV, HF as in
// march_pass).  ODD: the plane has an odd number of rows.
template <bool FIRST, bool LAST, bool EV, bool HF, bool ODD>
__device__ __forceinline__ void march3_pass(const FusedArgs &A, const March3Args &M, float kick, float drift,
                                            const ChainParams &prm, const Tile &tl, int chain,
                                            const float4 *tab, double *ksum, Totals *tot) {
    constexpr bool ACT = LAST || EV;
    const int P = A.g.P, nzs = M.nz, ny = A.g.nplanes, T = blockDim.x;
    // copy groups: plane z0 + it - 2 of psi (periodic) and plane it - 4 of p, two
    // iterations ahead (the slot freed by the plane that was central before)
    auto issue = [&](int it) {
        if (tl.rows > 0) {
            const int slot = it & (M3_RING - 1);
            int zw = M.z0 + it - 2;
            zw = zw < 0 ? zw + ny : zw;
            zw = zw >= ny ? zw - ny : zw;
            if (it < nzs + 4) {
                const float *s = M.src + (uint32_t)zw * (uint32_t)P;
                float *d = M.ring + slot * P;
                cp_async16(d + tl.e[0], s + tl.e[0]);
                if (!ODD || tl.rows == 2) cp_async16(d + tl.e[1], s + tl.e[1]);
            }
            if (!FIRST && it >= 4 && it < nzs + 4) {
                const float *s = M.p + (uint32_t)(M.z0 + it - 4) * (uint32_t)P;
                float *d = M.ring_p + slot * P;
                cp_async16(d + tl.e[0], s + tl.e[0]);
                if (!ODD || tl.rows == 2) cp_async16(d + tl.e[1], s + tl.e[1]);
            }
        }
        cp_commit();
    };
    const float hpf = kept(prm.hpf);
    float hrow[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i) hrow[i][0] = hrow[i][1] = hrow[i][2] = hrow[i][3] = hpf;
    auto load_field = [&](int z) {
        int zw = M.z0 + z;
        zw = zw < 0 ? zw + ny : zw;
        zw = zw < 0 ? zw + ny : zw;
        zw = zw >= ny ? zw - ny : zw;
        zw = zw >= ny ? zw - ny : zw;
        const float2 *hp = A.hdf + (uint32_t)zw * (uint32_t)P;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) hrow[i][k] = prm.betaf * hp[tl.e[i] + k].x;
    };
    if constexpr (HF) load_field(-3);
    const pair_t C2 = pk1(kept(prm.Cf)), bJ2 = pk1(kept(prm.bJf));
    const pair_t k2 = pk1(kick), d2 = pk1(drift);
    Window w[2];
    ActSums<1> as[2];
    AccRow<false> ks[2];
    ActPairs kc;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        w[i] = Window{row_zero(), row_zero(), row_zero(), row_zero()};
        if constexpr (ACT) as[i].clear();
        if constexpr (FIRST || LAST) ks[i].clear();
    }
    if constexpr (ACT) {
        const f2 cc = kept_df(prm.C), bj = kept_df(prm.bJ);
        kc.C = dup_df(cc);
        kc.bJ = dup_df(bj);
        kc.neg_C = pk1(-cc.hi);
        kc.neg_bJ = pk1(-bj.hi);
        kc.hp = dup_df(kept_df(prm.hp));
    }
    const uint32_t nz_own = tl.rows > 0 ? (uint32_t)nzs : 0u;

    auto step = [&](int it) {
        const int slot = it & (M3_RING - 1), cslot = (it - 1) & (M3_RING - 1), par = it & 1;
        cp_wait<1>();
        Row arr[2], pin[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            arr[i] = lds_row(M.ring + slot * P + tl.e[i]);
            pin[i] = FIRST ? row_zero() : lds_row(M.ring_p + slot * P + tl.e[i]);
        }
        __syncthreads();   // the last iteration's u and edges; the plane copied for it
        issue(it + 2);
        const int z = it - 3, zf = z - 1;   // plane of u; plane of the force
        const float2 *eb = M.edge + (par ^ 1) * 4 * T;   // [row][left end | right end][thread]
        const float *cp = M.ring + cslot * P;
        const Row ym = lds_row(cp + tl.ym), yp = lds_row(cp + tl.yp);
        const float *up = M.u + (par ^ 1) * P;
        const Row uym = lds_row(up + tl.ym), uyp = lds_row(up + tl.yp);
        Row un[2];
        float2 el[2], er[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            el[i] = eb[i * 2 * T + T + tl.left];
            er[i] = eb[i * 2 * T + tl.right];
        }
        // row i's neighbours in y: the other row of the tile and the row beyond
        // (a tile of one row has both beyond)
        const bool two = !ODD || tl.rows == 2;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            Window &v = w[i];
            const Row a = i == 0 ? ym : w[0].pc;
            const Row b = i == 1 ? yp : (two ? w[1].pc : yp);
            Row nb = x_sum<false>(v.pc, el[i].x, er[i].x, 4);
            nb = row_add(nb, row_add(a, b));
            nb = row_add(nb, row_add(v.pm, arr[i]));
            const pair_t ha = pk(hrow[i][0], hrow[i][1]), hb = pk(hrow[i][2], hrow[i][3]);
            const Row t{tanh2(fma2(C2, v.pc.a, fma2(bJ2, nb.a, ha))),
                        tanh2(fma2(C2, v.pc.b, fma2(bJ2, nb.b, hb)))};
            un[i] = Row{sub2(t.a, v.pc.a), sub2(t.b, v.pc.b)};
            if constexpr (ACT) {
                if ((uint32_t)z < nz_own && (i == 0 || two)) {
                    const uint32_t site0 = (uint32_t)(M.z0 + z) * (uint32_t)P + (uint32_t)tl.e[i];
                    const float4 sp = spin_u4(site0 >> 2, LAST ? M.traj : TRAJ_INIT, (uint32_t)chain,
                                              LAST ? A.round_keys : A.round_keys0);
                    const float su[4] = {sp.x, sp.y, sp.z, sp.w};
                    row_action<false, HF, 1, true>(A, prm, kc, v.pc, v.pm, arr[i], el[i].x, er[i].x, t, hrow[i],
                                                   4, site0, su, tab, as[i], &a, &b);
                }
            }
        }
        if constexpr (HF) load_field(z + 1);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            Window &v = w[i];
            const Row a = i == 0 ? uym : w[0].uc;
            const Row b = i == 1 ? uyp : (two ? w[1].uc : uyp);
            Row nu = x_sum<false>(v.uc, el[i].y, er[i].y, 4);
            nu = row_add(nu, row_add(a, b));
            nu = row_add(nu, row_add(v.um, un[i]));
            Row pv = pin[i];
            const bool inside = (uint32_t)zf < nz_own && (i == 0 || two);
            auto add_kinetic = [&](const Row &q) {
                f2 v0, v1, v2, v3;
                upk(half_square(q.a), v0, v1);
                upk(half_square(q.b), v2, v3);
                ks[i].add(v0);
                ks[i].add(v1);
                ks[i].add(v2);
                ks[i].add(v3);
            };
            const uint32_t o = (uint32_t)(M.z0 + zf) * (uint32_t)P + (uint32_t)tl.e[i];
            if constexpr (FIRST) {
                if (inside) {
                    const float4 g = momenta4(o >> 2, M.traj, (uint32_t)chain, A.round_keys);
                    pv = Row{pk(g.x, g.y), pk(g.z, g.w)};
                    add_kinetic(pv);
                }
            }
            pv.a = fma2(k2, fma2(C2, v.uc.a, mul2(bJ2, nu.a)), pv.a);
            pv.b = fma2(k2, fma2(C2, v.uc.b, mul2(bJ2, nu.b)), pv.b);
            if (inside) {
                *reinterpret_cast<ulonglong2 *>(M.p + o) = make_ulonglong2(pv.a, pv.b);
                if constexpr (!LAST)
                    *reinterpret_cast<ulonglong2 *>(M.dst + o) =
                        make_ulonglong2(fma2(d2, pv.a, v.pm.a), fma2(d2, pv.b, v.pm.b));
                else
                    add_kinetic(pv);
            }
        }
        // publish u and the row ends, move the windows on
        float *uo = M.u + par * P;
        float2 *ew = M.edge + par * 4 * T + tl.tid;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (tl.rows > i) sts_row(uo + tl.e[i], un[i]);
            float f0, f1, f2_, f3, u0, u1, u2, u3;
            upk(arr[i].a, f0, f1); upk(arr[i].b, f2_, f3);
            upk(un[i].a, u0, u1); upk(un[i].b, u2, u3);
            ew[i * 2 * T] = make_float2(f0, u0);
            ew[i * 2 * T + T] = make_float2(f3, u3);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            w[i].pm = w[i].pc;
            w[i].pc = arr[i];
            w[i].um = w[i].uc;
            w[i].uc = un[i];
        }
    };
    issue(0);
    issue(1);
    const int n_it = nzs + 4;   // output plane it - 4
    if constexpr (FIRST || LAST) {
        // their loop body is long (draws, action): once, with moves between the
        // windows' registers, instead of three times (instruction fetch was the
        // longest stall: 0.47 ms for the two sweeps at 608 chains of L = 32)
#pragma unroll 1
        for (int it = 0; it < n_it; ++it) step(it);
    } else {
#pragma unroll 1
        for (int it = 0; it < n_it; it += 3) {   // (planes past the end are computed and dropped)
            step(it);
            step(it + 1);
            step(it + 2);
        }
    }
    cp_wait<0>();
    __syncthreads();
    if constexpr (FIRST || LAST) *ksum = ks[0].value() + ks[1].value();
    if constexpr (ACT) {
        tot->S = tot->T = tot->AT = tot->HT = 0.0;
        tot->sS = 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            tot->S += as[i].S.value();
            tot->sS += as[i].sS;
            tot->T += kahan_val(as[i].sT[0], as[i].cT[0]);
            tot->AT += kahan_val(as[i].sAT[0], as[i].cAT[0]);
            tot->HT += kahan_val(as[i].sHT[0], as[i].cHT[0]);
        }
    }
}

// One CTA, or (CL) one cluster of A.cs CTAs, per chain.
template <bool CL, bool HF, bool ODD>
__global__ void __launch_bounds__(M3_THREADS, 1)
    march3_kernel(const __grid_constant__ FusedArgs A, const __grid_constant__ Schedule S) {
    extern __shared__ float4 smem_f4[];
    const Geometry &g = A.g;
    const int T = blockDim.x;
    for (int i = threadIdx.x; i < LOG1PEXP_NODES; i += T) smem_f4[i] = A.lpe_tab[i];
    const float4 *tab = smem_f4;
    March3Args M;
    M.ring = reinterpret_cast<float *>(smem_f4 + LOG1PEXP_NODES);
    M.ring_p = M.ring + M3_RING * g.P;
    M.u = M.ring_p + M3_RING * g.P;
    M.edge = reinterpret_cast<float2 *>(M.u + 2 * g.P);
    double *red = reinterpret_cast<double *>(M.edge + 8 * T);
    int *bcast = reinterpret_cast<int *>(red + 32 * 8);
    double *xch = red + 32 * 8 + 2;        // two exchange buffers of XCH_WORDS
    double *k0 = xch + 2 * XCH_WORDS;      // the trajectory's K0, S of the start (thread 0)
    const int cs = CL ? cluster_size() : 1, cr = CL ? cluster_rank() : 0;
    const int chain = A.chain0 + (int)(blockIdx.x / (unsigned)cs);
    if (chain >= A.n_chains) return;   // uniform over the cluster
    const bool lead = cr == 0;
    if (CL && cs != A.cs && lead && threadIdx.x == 0) atomicOr(A.err, KERR_BOUNDS);
    ChainState *const st = A.state + chain;
    const ChainParams &prm = A.params[chain];
    const Tile tl = make_tile(g);
    M.z0 = (int)((int64_t)cr * g.nplanes / cs);
    M.nz = (int)((int64_t)(cr + 1) * g.nplanes / cs) - M.z0;
    const int64_t cbase = (int64_t)chain * g.N;
    M.p = A.p + cbase;
    // what the slab reads before it is written: the ring's rows of a one-row
    // tile, the first edge values
    for (int i = threadIdx.x; i < (2 * M3_RING + 2) * g.P; i += T) M.ring[i] = 0.0f;
    for (int i = threadIdx.x; i < 8 * T; i += T) M.edge[i] = make_float2(0.0f, 0.0f);
    __syncthreads();
    int start = st->start;
    if (threadIdx.x == 0) k0[1] = st->S;
    auto pass_end = [&]() {
        if (CL && cs > 1) cluster_barrier();   // the neighbours' planes are read and rewritten next
    };
    for (int k = 0; k < A.n_traj; ++k) {
        const uint32_t traj = A.traj0 + (uint32_t)k;
        M.traj = traj;
        int src = start, dst = (start + 1) % 3;
        auto buffers = [&]() {
            M.src = sel3(A, src) + cbase;
            M.dst = sel3(A, dst) + cbase;
        };
        auto advance = [&]() {
            const int was = src;
            src = dst;
            dst = was == start ? (start + 2) % 3 : was;
        };
        auto kk = [&](int j) { return kept((float)(S.kick[j] * prm.eps)); };
        auto dd = [&](int j) { return kept((float)(S.drift[j] * prm.eps)); };
        buffers();
        double v1[1];
        if (k == 0 && A.eval_start) {
            Totals ini;
            march3_pass<true, false, true, HF, ODD>(A, M, kk(0), dd(0), prm, tl, chain, tab, v1, &ini);
            pass_end();
            double ev[5] = {ini.S, ini.T, ini.AT, ini.HT, (double)ini.sS};
            chain_sum<5, CL>(ev, red, xch + XCH_WORDS, cs);
            if (threadIdx.x == 0) {
                k0[1] = ev[0];
                if (lead) {
                    st->S = ev[0];
                    set_obs(st, prm, ev[1], ev[2], ev[3], ev[4], 1.0 / (double)g.N);
                    st->prop = start;
                }
            }
        } else {
            march3_pass<true, false, false, HF, ODD>(A, M, kk(0), dd(0), prm, tl, chain, tab, v1, nullptr);
            pass_end();
        }
        block_sum<1>(v1, red);   // this CTA's K0
        if (threadIdx.x == 0) k0[0] = v1[0];
        advance();
        for (int j = 1; j + 1 < S.n_pass; ++j) {
            buffers();
            march3_pass<false, false, false, HF, ODD>(A, M, kk(j), dd(j), prm, tl, chain, tab, nullptr, nullptr);
            pass_end();
            advance();
        }
        buffers();
        const int prop = src;   // the last evaluation writes no psi
        Totals end;
        march3_pass<false, true, false, HF, ODD>(A, M, kk(S.n_pass - 1), 0.0f, prm, tl, chain, tab, v1, &end);
        pass_end();
        const double invN = 1.0 / (double)g.N;
        double v[7] = {threadIdx.x == 0 ? k0[0] : 0.0, v1[0], end.S, end.T, end.AT, end.HT, (double)end.sS};
        chain_sum<7, CL>(v, red, xch, cs);
        double S_cur = threadIdx.x == 0 ? k0[1] : 0.0;
        start = metropolis_step(CtaThreads{}, A, st, prm, chain, traj, start, prop, v, invN, S_cur, lead, bcast);
        if (A.flip_every > 0 && ((traj + 1) % (uint32_t)A.flip_every) == 0) {
            Acc fa = acc_zero();
            action_sweep<3, 4, CL>(A, prm, chain, start, -1.0f, traj, A.seed, make_slots<4>(g, threadIdx.x, T),
                                   tab, fa, M.z0, M.z0 + M.nz);
            double wv[5] = {acc_val(fa.S, fa.Slo), kahan_val(fa.sT, fa.cT), kahan_val(fa.sAT, fa.cAT),
                            kahan_val(fa.sHT, fa.cHT), (double)fa.sS};
            chain_sum<5, CL>(wv, red, xch + XCH_WORDS, cs);
            if (flip_step(CtaThreads{}, A, st, prm, chain, traj, wv, invN, S_cur, lead, bcast)) {
                const int f = (start != prop) ? 3 - start - prop : (start + 1) % 3;
                const int64_t off = cbase + (int64_t)M.z0 * g.P, cnt = (int64_t)M.nz * g.P;
                const float *gs = sel3(A, start) + off;
                float *gf = sel3(A, f) + off;
                for (int64_t i = threadIdx.x; i < cnt; i += T) gf[i] = -gs[i];
                start = f;
                if (threadIdx.x == 0 && lead) st->start = f;
                pass_end();
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) k0[1] = S_cur;
        measure_step(CtaThreads{}, A, st, traj, lead);
    }
    if (CL && cs > 1) cluster_barrier();   // no CTA leaves while its exchange buffers may be read
}

template <bool CL, bool HF, bool ODD>
cudaError_t node3(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    auto kern = march3_kernel<CL, HF, ODD>;
    static DeviceOnce once;
    const cudaError_t e = allow_smem(once, kern, 227 * 1024);
    if (e != cudaSuccess) return e;
    np->func = reinterpret_cast<void *>(kern);
    np->gridDim = dim3((unsigned)((a.n_chains - a.chain0) * a.cs), 1, 1);
    np->blockDim = dim3((unsigned)a.march, 1, 1);
    np->sharedMemBytes = (unsigned)m3_smem(a.g.P, a.march);
    np->kernelParams = args;
    np->extra = nullptr;
    return cudaSuccess;
}

}  // namespace

// Kernel-node parameters (one translation unit without and one with a field).
cudaError_t march3_node_plain(const FusedArgs &a, cudaKernelNodeParams *np, void **args);
cudaError_t march3_node_field(const FusedArgs &a, cudaKernelNodeParams *np, void **args);

}  // namespace ihmc
