// march_lattice.cuh -- FP32 HMC trajectories on 2D lattices, several force
// evaluations per sweep over the chain.
//
// The plane-streaming kernel (fused_lattice_impl.cuh) moves psi and p through
// HBM once per force evaluation (16 B per site-step) and spends more than half
// of its instructions on ring addresses and shared-memory neighbour loads.
// Here a thread owns four consecutive columns and marches down the rows with
// its own three-row windows of psi and u in registers, so the neighbours along
// the march need no load at all; the neighbours in the row come from the
// threads left and right, which publish the end values of their four columns
// in shared memory (two 8-byte stores, two 8-byte loads per evaluation).
//
// K consecutive force evaluations of the integrator run in one sweep as a
// pipeline: evaluation s works two rows behind evaluation s - 1, whose output
// rows are its input rows and never leave the registers.  psi and p then
// cross HBM once per K evaluations.  One barrier per row serves all K.
//
// Periodic wrap: evaluation s needs rows beyond both ends of the chain, so
// the sweep recomputes 2 (K - s) rows at either end instead of keeping them:
// input rows -2K .. nz + 2K - 1, output rows 0 .. nz - 1.  psi is read from
// one buffer and written to another, so its first rows are still the old ones
// at the end of the sweep; p is updated in place, so the old p of the first
// 2K - 2 rows is kept in shared memory (each thread its own columns).
//
// Why three: one trajectory of 1216 chains of L = 1024, N_md = 20, took 82.5 ms
// on the plane-streaming kernel (21 sweeps, 4.9 TB/s, 87 instructions per
// site and evaluation).  Here 71 ms with one evaluation per sweep (memory-bound:
// 2.9 ms a sweep), 41 ms with two, 33.8 ms with three (3.3 ms a sweep, 22
// instructions per site and evaluation, at the copy rate again), 43 ms with four
// (over 128 registers, so half the warps).  The first and the last sweep, with
// the draws and the action, take 13 ms of it and are bound by issue (60 % of the
// slots) and the FP32 pipe.  L = 256: 5.9 -> 2.15 ms.
//
// A chain whose rows fill only part of a CTA can be cut into slabs of rows, one
// per group of threads (few chains, which would leave the SMs without warps).
//
// Registers: 128 a thread (two CTAs of 256 threads on an SM) are fewer than the three
// evaluations want.  The compiler spills 116 .. 144 bytes a thread (stores; loads 156 ..
// 256) for rows of whole vectors, 320 .. 404 (448 .. 588) with a field per site, and for
// ragged rows, whose draws and masks come on top, 1204 .. 1368 (1640 .. 1856), with a
// field 1808 .. 1820 (1884 .. 1924): the reason that march_lattice_pays leaves many of
// those to the plane-streaming kernel.
//
// Every value is computed by the operations of the plane-streaming kernel in
// the same order (the packed FP32 pair instructions round each half exactly as
// the scalar ones do): psi and p agree bit for bit, and so do the per-thread
// partial sums of the energies where a thread has the same columns in both.
#pragma once
#include "fused_lattice_impl.cuh"
#include "pair.cuh"

namespace ihmc {
namespace {

// Four consecutive columns of one row.
struct Row {
    pair_t a, b;
};
__device__ __forceinline__ Row row_zero() { return Row{0ull, 0ull}; }
__device__ __forceinline__ Row lds_row(const float *p) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
    return Row{t.x, t.y};
}
__device__ __forceinline__ void sts_row(float *p, const Row &r) {
    *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(r.a, r.b);
}

constexpr int MARCH_K = 3;             // evaluations per sweep between the ends of a trajectory
constexpr int MARCH_MIN_SLAB = 24;     // rows
constexpr int MARCH_SLOTS = 3;         // rows of psi and p in flight per thread, and edge buffers
constexpr int MARCH_CTA_THREADS = 256;   // at most: 128 registers a thread, two CTAs per SM

// Shared memory of one slab (floats), TS threads' worth, up to K evaluations
// per sweep: psi and p rows in flight, edge values, old p of the rows beyond
// its end and, where the chain is cut into slabs, of those before its start.
__host__ __device__ constexpr int march_floats(int TS, int K, bool cut) {
    return TS * (2 * 4 * MARCH_SLOTS + MARCH_SLOTS * K * 4 + (2 * K - 2) * (cut ? 2 : 1) * 4);
}
// Reduction words of one chain: 8 warps of 8 doubles, two broadcast words, K0.
constexpr int MARCH_RED_BYTES = 8 * 8 * 8 + 32;

// Threads that work on a slab or on a chain (a multiple of 32), with a barrier
// of their own: several chains with short rows share a CTA, and with it the
// table of the action, or several slabs of one chain do.
struct ChainThreads {
    int tid, T, id;
    __device__ __forceinline__ bool first() const { return tid == 0; }
    __device__ __forceinline__ void sync() const {
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(T) : "memory");
    }
};

// block_sum (device_common.cuh) over the threads of one chain.
template <int NV>
__device__ __forceinline__ void chain_threads_sum(double (&v)[NV], double *scratch, const ChainThreads &th) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
    }
    const int warp = th.tid >> 5, lane = th.tid & 31;
    th.sync();
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) scratch[warp * NV + k] = v[k];
    }
    th.sync();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double s = 0.0;
        for (int w = 0; w < th.T >> 5; ++w) s += scratch[w * NV + k];
        v[k] = s;
    }
    th.sync();
}

// What a thread keeps for the whole launch: its first column, how many of its
// four columns exist (0: an idle thread of the last warp) and its neighbours.
struct Cols {
    int e0, m, left, right;
};
__device__ __forceinline__ Cols make_cols(int X, int t) {
    const int nvec = (X + 3) >> 2;
    Cols c;
    c.m = t < nvec ? (X - 4 * t < 4 ? X - 4 * t : 4) : 0;
    c.e0 = t < nvec ? 4 * t : 0;
    c.left = t < nvec ? (t == 0 ? nvec - 1 : t - 1) : t;
    c.right = t < nvec ? (t == nvec - 1 ? 0 : t + 1) : t;
    return c;
}

// Left and right neighbours of the four columns.  RAG: the last thread may own
// fewer than four; its last existing column's right neighbour is rx as well.
template <bool RAG>
__device__ __forceinline__ void x_neighbours(const Row &c, float lw, float rx, int m, float (&l)[4],
                                             float (&r)[4]) {
    float c0, c1, c2, c3;
    upk(c.a, c0, c1);
    upk(c.b, c2, c3);
    l[0] = lw; l[1] = c0; l[2] = c1; l[3] = c2;
    r[0] = c1; r[1] = c2; r[2] = c3; r[3] = rx;
    if constexpr (RAG) {
#pragma unroll
        for (int k = 0; k < 3; ++k) r[k] = m == k + 1 ? rx : r[k];
    }
}
template <bool RAG>
__device__ __forceinline__ Row x_sum(const Row &c, float lw, float rx, int m) {
    float l[4], r[4];
    x_neighbours<RAG>(c, lw, rx, m, l, r);
    return Row{pk(l[0] + r[0], l[1] + r[1]), pk(l[2] + r[2], l[3] + r[3])};
}
// The last existing column's value (published to the right-hand neighbour).
template <bool RAG>
__device__ __forceinline__ float last_col(const Row &c, int m) {
    float c0, c1, c2, c3;
    upk(c.a, c0, c1);
    upk(c.b, c2, c3);
    if constexpr (RAG) return m == 4 ? c3 : m == 3 ? c2 : m == 2 ? c1 : c0;
    return c3;
}

// Per-chain constants of the action as pairs, kept in registers.
struct ActPairs {
    f2x2 C, bJ, hp;
    pair_t neg_C, neg_bJ;
};
__device__ __forceinline__ f2 kept_df(double x) {
    const f2 v = df_from_double(x);
    return f2{kept(v.hi), kept(v.lo)};
}

// Sums of one evaluation of the action (or of K0) over a thread's columns.
// Estimators: Kahan FP32 sums, one set per column where rows are scalar (RAG:
// Kahan's scheme rounds every addend by up to half an ulp, so the columns stay
// apart as in the plane-streaming kernel, whose threads own one column), else
// one set of the sums over four columns.
template <int NE>
struct ActSums {
    AccRow<(NE > 1)> S;
    float sT[NE], cT[NE], sAT[NE], cAT[NE], sHT[NE], cHT[NE];
    int sS;
    __device__ __forceinline__ void clear() {
        S.clear();
        sS = 0;
#pragma unroll
        for (int k = 0; k < NE; ++k) sT[k] = cT[k] = sAT[k] = cAT[k] = sHT[k] = cHT[k] = 0.0f;
    }
};
struct Totals {
    double S, T, AT, HT;
    int sS;
};

// Action terms of four sites (vector_action's formulas and values) in pair
// arithmetic, the estimators and the conditional spin draws.  ym, yp: the rows
// before and after in the plane (3D, else null).
template <bool RAG, bool HF, int NE, bool D3 = false>
__device__ __forceinline__ void row_action(const FusedArgs &A, const ChainParams &prm, const ActPairs &kc,
                                           const Row &c, const Row &zm, const Row &zp, float lw, float rx,
                                           const Row &t, const float (&hf)[4], int m, uint32_t site0,
                                           const float (&su)[4], const float4 *tab, ActSums<NE> &ac,
                                           const Row *ym = nullptr, const Row *yp = nullptr) {
    float l[4], r[4];
    x_neighbours<RAG>(c, lw, rx, m, l, r);
    const bool has_h = HF || prm.hp != 0.0;
    f2x2 si[2];
    float ahi[4], tv[4];
    upk(t.a, tv[0], tv[1]);
    upk(t.b, tv[2], tv[3]);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const pair_t ps = q ? c.b : c.a;
        f2x2 nb = two_sum(pk(l[2 * q], l[2 * q + 1]), pk(r[2 * q], r[2 * q + 1]));
        if constexpr (D3) {
            nb = df_add_f(nb, q ? ym->b : ym->a);
            nb = df_add_f(nb, q ? yp->b : yp->a);
        }
        nb = df_add_f(nb, q ? zm.b : zm.a);
        nb = df_add_f(nb, q ? zp.b : zp.a);
        const f2x2 a = df_add_q(df_mul_fc(kc.C, kc.neg_C, ps), df_mul(kc.bJ, kc.neg_bJ, nb));
        f2x2 x = a;
        if constexpr (HF) {
            const f2 b2 = df_from_double(prm.beta);
            f2 h0{0.0f, 0.0f}, h1{0.0f, 0.0f};
            if (!RAG || 2 * q < m) {
                const float2 v = A.hdf[site0 + 2 * q];
                h0 = df_mul(b2, f2{v.x, v.y});
            }
            if (!RAG || 2 * q + 1 < m) {
                const float2 v = A.hdf[site0 + 2 * q + 1];
                h1 = df_mul(b2, f2{v.x, v.y});
            }
            x = df_add_q(a, f2x2{pk(h0.hi, h1.hi), pk(h0.lo, h1.lo)});
        } else if (has_h) {
            x = df_add_q(a, kc.hp);
        }
        si[q] = action_term(ps, a, x, tab);
        upk(a.hi, ahi[2 * q], ahi[2 * q + 1]);
    }
    if constexpr (RAG) {   // columns that do not exist add nothing
        float v[4], w[4];
        upk(si[0].hi, v[0], v[1]); upk(si[1].hi, v[2], v[3]);
        upk(si[0].lo, w[0], w[1]); upk(si[1].lo, w[2], w[3]);
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            v[k] = k < m ? v[k] : 0.0f;
            w[k] = k < m ? w[k] : 0.0f;
        }
        si[0] = f2x2{pk(v[0], v[1]), pk(w[0], w[1])};
        si[1] = f2x2{pk(v[2], v[3]), pk(w[2], w[3])};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k >= m) break;
            kahan_add(ac.sT[k % NE], ac.cT[k % NE], tv[k]);
            kahan_add(ac.sAT[k % NE], ac.cAT[k % NE], ahi[k] * tv[k]);
            if (has_h) kahan_add(ac.sHT[k % NE], ac.cHT[k % NE], hf[k] * tv[k]);
        }
    } else {
        float vT = 0.0f, vAT = 0.0f, vHT = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            vT += tv[k];
            vAT = fmaf(ahi[k], tv[k], vAT);
            if (has_h) vHT = fmaf(hf[k], tv[k], vHT);
        }
        kahan_add(ac.sT[0], ac.cT[0], vT);
        kahan_add(ac.sAT[0], ac.cAT[0], vAT);
        if (has_h) kahan_add(ac.sHT[0], ac.cHT[0], vHT);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (!RAG || k < m) ac.sS += (su[k] < (1.0f + tv[k]) * 0.5f) ? 1 : -1;
    if constexpr (RAG) {
        ac.S.add(si[0], si[1]);
    } else {
        f2 v0, v1, v2, v3;
        upk(si[0], v0, v1);
        upk(si[1], v2, v3);
        ac.S.add(df_add_q(df_add_q(df_add_q(v0, v1), v2), v3));
    }
}

// One evaluation's window: rows z - 1, z of psi and z - 2, z - 1 of u on entry
// of the iteration in which row z + 1 of psi arrives.
struct Window {
    Row pm, pc, um, uc;
};

struct MarchArgs {
    int z0, nz;          // the slab's rows: z0 .. z0 + nz - 1
    const float *src;    // psi read (chain base)
    float *dst, *p;      // psi written, momenta (chain base)
    uint32_t traj;
    float *ring;         // this thread's part of the rows in flight
    float2 *edge;        // edge values: [slot][evaluation][left end | right end][thread]
    float *old_p;        // old p beyond the slab's end (and before it), this thread's columns
};

// K force evaluations over all rows of the chain.  kick and drift: already
// times eps.  FIRST: evaluation 0 is the trajectory's first (draws the momenta;
// ksum gets K0; EV: also the action of the configuration read, into *tot); LAST:
// evaluation K - 1 is its last (no drift; ksum gets K1, *tot the action of the
// proposal, which dst receives).  HF: a
// field per site.  TS: the row stride of the shared arrays, in threads (known
// to the compiler: the shared addresses are then offsets of a few registers).
template <int TS, bool CUT, int K, bool FIRST, bool LAST, bool EV, bool RAG, bool HF>
__device__ __forceinline__ void march_pass(const FusedArgs &A, const MarchArgs &M, const ChainThreads &th,
                                           const float (&kick)[K], const float (&drift)[K],
                                           const ChainParams &prm, const Cols &cl, int chain,
                                           const float4 *tab, double *ksum, Totals *tot) {
    constexpr bool ACT = LAST || EV;
    constexpr int NE = RAG ? 4 : 1;
    const int X = A.g.X, ny = A.g.nplanes, tid = th.tid;
    const int z0 = CUT ? M.z0 : 0, nz = CUT ? M.nz : ny;   // the slab's rows
    float *ring_p = M.ring + MARCH_SLOTS * 4 * TS;

    // Rows are issued in order, three iterations ahead: arriving row it - 2K
    // (periodic) of psi and the row two before it of p.  A thread copies and
    // reads only its own columns.  Every iteration copies both (rows that no
    // evaluation uses are in range too): offsets advance by one wrapped add.
    const uint32_t N32 = (uint32_t)A.g.N, X32 = (uint32_t)X;   // sites per chain <= 2^31
    uint32_t o_psi, o_p;
    {
        int r = z0 - 2 * K, rp = z0 - 2 * K - 2;
        while (r < 0) r += ny;
        while (rp < 0) rp += ny;
        o_psi = (uint32_t)r * X32;
        o_p = (uint32_t)rp * X32;
    }
    const float *g_psi = M.src + cl.e0;
    float *g_p = M.p + cl.e0;
    float *g_dst = M.dst + cl.e0;
    auto copy_row = [&](float *d, const float *s) {
        if constexpr (!RAG) {
            if (cl.m > 0) cp_async16(d, s);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < cl.m) cp_async4(d + k, s + k);
        }
    };
    auto wrap_add = [&](uint32_t o) {   // o + X modulo N
        const uint32_t a = o + X32;
        return min(a, a - N32);
    };
    auto issue = [&](int slot) {
        copy_row(M.ring + slot * 4 * TS, g_psi + o_psi);
        if constexpr (!FIRST) copy_row(ring_p + slot * 4 * TS, g_p + o_p);
        cp_commit();
        o_psi = wrap_add(o_psi);
        o_p = wrap_add(o_p);
    };
    const uint32_t nz_own = cl.m > 0 ? (uint32_t)nz : 0u;   // rows this thread stores and counts

    // per-site field of evaluation s at its row z, loaded one iteration ahead
    float hrow[HF ? K : 1][4];
    const float hpf = kept(prm.hpf);
    if constexpr (!HF) hrow[0][0] = hrow[0][1] = hrow[0][2] = hrow[0][3] = hpf;
    auto load_field = [&](int z, float (&h)[4]) {
        int zw = z0 + z;
        while (zw < 0) zw += ny;
        while (zw >= ny) zw -= ny;
        const float2 *hp = A.hdf + ((uint32_t)zw * X32 + (uint32_t)cl.e0);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            h[k] = (!RAG || k < cl.m) ? prm.betaf * hp[k].x : 0.0f;
    };

    Window w[K];
    Row dly[K > 1 ? K - 1 : 1][2];   // kicked momenta on their way to the next evaluation
#pragma unroll
    for (int s = 0; s < K; ++s) w[s] = Window{row_zero(), row_zero(), row_zero(), row_zero()};
#pragma unroll
    for (int s = 0; s + 1 < K; ++s) dly[s][0] = dly[s][1] = row_zero();
    if constexpr (HF) {
#pragma unroll
        for (int s = 0; s < K; ++s) load_field(-2 * K - 1 - 2 * s, hrow[s]);
    }

    const pair_t C2 = pk1(kept(prm.Cf)), bJ2 = pk1(kept(prm.bJf)), hp2 = pk1(hpf);
    ActPairs kc;
    ActSums<NE> as;
    AccRow<RAG> ks;
    if constexpr (FIRST || LAST) ks.clear();
    if constexpr (ACT) {
        const f2 cc = kept_df(prm.C), bj = kept_df(prm.bJ);
        kc.C = dup_df(cc);
        kc.bJ = dup_df(bj);
        kc.neg_C = pk1(-cc.hi);
        kc.neg_bJ = pk1(-bj.hi);
        kc.hp = dup_df(kept_df(prm.hp));
        as.clear();
    }

    // slot: of the row arriving now; prev: edge buffer of the last iteration
    auto step = [&](int it, int slot, int prev) {
        cp_wait<MARCH_SLOTS - 1>();
        Row arr = lds_row(M.ring + slot * 4 * TS);
        Row pin = FIRST ? row_zero() : lds_row(ring_p + slot * 4 * TS);
        th.sync();   // the edge values of the last iteration; the slot is free again
        issue(slot);
        if constexpr (K > 1 && !FIRST) {
            const int rp = it - 2 * K - 2;
            if (!CUT && (unsigned)rp < (unsigned)(2 * K - 2)) sts_row(M.old_p + rp * 4 * TS, pin);
            if ((unsigned)(rp - nz) < (unsigned)(2 * K - 2)) pin = lds_row(M.old_p + (rp - nz) * 4 * TS);
            if constexpr (CUT) {   // before the slab's start
                if ((unsigned)(rp + 2 * K - 2) < (unsigned)(2 * K - 2))
                    pin = lds_row(M.old_p + (rp + 4 * K - 4) * 4 * TS);
            }
        }
#pragma unroll
        for (int s = 0; s < K; ++s) {
            Window &v = w[s];
            const int z = it - 2 * K - 1 - 2 * s;   // row of u; the force is for row z - 1
            const float2 *eb = M.edge + (prev * K + s) * 2 * TS;
            const float2 el = eb[TS + cl.left], er = eb[cl.right];   // {psi, u}
            // ---- u(z) = tanh(A psi + h') - psi ----
            Row nb = x_sum<RAG>(v.pc, el.x, er.x, cl.m);
            nb.a = add2(nb.a, add2(v.pm.a, arr.a));
            nb.b = add2(nb.b, add2(v.pm.b, arr.b));
            pair_t ha = hp2, hb = hp2;
            if constexpr (HF) {
                ha = pk(hrow[s][0], hrow[s][1]);
                hb = pk(hrow[s][2], hrow[s][3]);
            }
            const Row t{tanh2(fma2(C2, v.pc.a, fma2(bJ2, nb.a, ha))),
                        tanh2(fma2(C2, v.pc.b, fma2(bJ2, nb.b, hb)))};
            const Row un{sub2(t.a, v.pc.a), sub2(t.b, v.pc.b)};
            if constexpr (ACT) {
                if (s == (LAST ? K - 1 : 0) && (uint32_t)z < nz_own) {
                    const uint32_t st = LAST ? M.traj : TRAJ_INIT;
                    const uint32_t *rk = LAST ? A.round_keys : A.round_keys0;
                    const uint32_t site0 = (uint32_t)(z0 + z) * X32 + (uint32_t)cl.e0;
                    float su[4];
                    if constexpr (!RAG) {
                        const float4 g = spin_u4(site0 >> 2, st, (uint32_t)chain, rk);
                        su[0] = g.x; su[1] = g.y; su[2] = g.z; su[3] = g.w;
                    } else {
                        // rows start anywhere in the groups of four sites that
                        // share a random block: two blocks cover the columns
                        spin_u4_any(site0, st, (uint32_t)chain, rk, su);
                    }
                    row_action<RAG, HF>(A, prm, kc, v.pc, v.pm, arr, el.x, er.x, t, hrow[HF ? s : 0], cl.m, site0, su,
                                        tab, as);
                }
            }
            if constexpr (HF) load_field(z + 1, hrow[s]);
            // ---- F(z - 1) = A u, kick, drift ----
            const int zf = z - 1;
            Row nu = x_sum<RAG>(v.uc, el.y, er.y, cl.m);
            nu.a = add2(nu.a, add2(v.um.a, un.a));
            nu.b = add2(nu.b, add2(v.um.b, un.b));
            Row pv = pin;
            const bool inside = (uint32_t)zf < nz_own;
            auto add_kinetic = [&](const Row &q) {
                f2x2 ha = half_square(q.a), hb = half_square(q.b);
                if constexpr (RAG) {
                    float v4[4], w4[4];
                    upk(ha.hi, v4[0], v4[1]); upk(hb.hi, v4[2], v4[3]);
                    upk(ha.lo, w4[0], w4[1]); upk(hb.lo, w4[2], w4[3]);
#pragma unroll
                    for (int k = 1; k < 4; ++k) {
                        v4[k] = k < cl.m ? v4[k] : 0.0f;
                        w4[k] = k < cl.m ? w4[k] : 0.0f;
                    }
                    ha = f2x2{pk(v4[0], v4[1]), pk(w4[0], w4[1])};
                    hb = f2x2{pk(v4[2], v4[3]), pk(w4[2], w4[3])};
                }
                if constexpr (RAG) {
                    ks.add(ha, hb);
                } else {
                    f2 v0, v1, v2, v3;
                    upk(ha, v0, v1);
                    upk(hb, v2, v3);
                    ks.add(v0);
                    ks.add(v1);
                    ks.add(v2);
                    ks.add(v3);
                }
            };
            if constexpr (FIRST) {
                // the rows beyond the ends, which later evaluations of the
                // sweep need, draw their momenta again
                if (s == 0 && cl.m > 0 && zf > -2 * K + 1 && zf < nz + 2 * K - 2) {
                    float z4[4];
                    int zw = z0 + zf;
                    if constexpr (K > 1) zw = zw < 0 ? zw + ny : zw >= ny ? zw - ny : zw;
                    const uint32_t site0 = (uint32_t)zw * X32 + (uint32_t)cl.e0;
                    if constexpr (!RAG) {
                        const float4 g = momenta4(site0 >> 2, M.traj, (uint32_t)chain, A.round_keys);
                        z4[0] = g.x; z4[1] = g.y; z4[2] = g.z; z4[3] = g.w;
                    } else {
                        momenta4_any(site0, M.traj, (uint32_t)chain, A.round_keys, z4);
                    }
                    pv = Row{pk(z4[0], z4[1]), pk(z4[2], z4[3])};
                    if (inside) add_kinetic(pv);
                }
            }
            const pair_t k2 = pk1(kick[s]);
            pv.a = fma2(k2, fma2(C2, v.uc.a, mul2(bJ2, nu.a)), pv.a);
            pv.b = fma2(k2, fma2(C2, v.uc.b, mul2(bJ2, nu.b)), pv.b);
            Row pn = row_zero();   // drifted psi row z - 1
            const bool drifts = !LAST || s + 1 < K;
            if (drifts) {
                const pair_t d2 = pk1(drift[s]);
                pn = Row{fma2(d2, pv.a, v.pm.a), fma2(d2, pv.b, v.pm.b)};
            } else if (inside) {
                add_kinetic(pv);
            }
            // p leaves with the last evaluation, psi with the last drift
            const bool store_p = s == K - 1, store_psi = s == (LAST ? K - 2 : K - 1);
            if ((store_p || store_psi) && inside) {
                const uint32_t o = (uint32_t)(z0 + zf) * X32;
                if constexpr (!RAG) {
                    if (store_p) *reinterpret_cast<ulonglong2 *>(g_p + o) = make_ulonglong2(pv.a, pv.b);
                    if (store_psi) *reinterpret_cast<ulonglong2 *>(g_dst + o) = make_ulonglong2(pn.a, pn.b);
                } else {
                    float q[4], x[4];
                    upk(pv.a, q[0], q[1]); upk(pv.b, q[2], q[3]);
                    upk(pn.a, x[0], x[1]); upk(pn.b, x[2], x[3]);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k < cl.m) {
                            if (store_p) g_p[o + k] = q[k];
                            if (store_psi) g_dst[o + k] = x[k];
                        }
                }
            }
            // ---- publish the row ends, move the windows on ----
            {
                float f0, f1, u0, u1;
                upk(arr.a, f0, f1);
                upk(un.a, u0, u1);
                float2 *ew = M.edge + (slot * K + s) * 2 * TS + tid;
                ew[0] = make_float2(f0, u0);
                ew[TS] = make_float2(last_col<RAG>(arr, cl.m), last_col<RAG>(un, cl.m));
            }
            v.pm = v.pc;
            v.pc = arr;
            v.um = v.uc;
            v.uc = un;
            if (s + 1 < K) {
                pin = dly[s][0];
                dly[s][0] = dly[s][1];
                dly[s][1] = pv;
                arr = pn;
            }
        }
    };

    // the neighbouring slabs update the rows beyond this one's ends in place:
    // their old p is kept before any slab starts
    if constexpr (K > 1 && !FIRST && CUT) {
        for (int i = 0; i < 4 * K - 4; ++i) {
            int row = i < 2 * K - 2 ? z0 + nz + i : z0 + i - (4 * K - 4);
            row = row < 0 ? row + ny : row >= ny ? row - ny : row;
            copy_row(M.old_p + i * 4 * TS, g_p + (uint32_t)row * X32);
        }
        cp_commit();
        cp_wait<0>();
        __syncthreads();
    }
    // edge buffer 2 is read by the first iteration (before anything valid)
    for (int s = 0; s < 2 * K; ++s) M.edge[(2 * K * 2 + s) * TS + tid] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int it = 0; it < MARCH_SLOTS; ++it) issue(it);
    const int n_it = nz + 4 * K;   // output row it - 4K
#pragma unroll 1
    for (int it = 0; it < n_it; it += 3) {   // (rows past the end are computed and dropped)
        step(it, 0, 2);
        step(it + 1, 1, 0);
        step(it + 2, 2, 1);
    }
    cp_wait<0>();
    if constexpr (CUT) __syncthreads();   // the other slabs' rows are written
    else th.sync();
    if constexpr (FIRST || LAST) *ksum = ks.value();
    if constexpr (ACT) {
        tot->S = as.S.value();
        tot->sS = as.sS;
        tot->T = tot->AT = tot->HT = 0.0;
#pragma unroll
        for (int k = 0; k < NE; ++k) {
            tot->T += kahan_val(as.sT[k], as.cT[k]);
            tot->AT += kahan_val(as.sAT[k], as.cAT[k]);
            tot->HT += kahan_val(as.sHT[k], as.cHT[k]);
        }
    }
}

// T = A.march threads per chain, blockDim.x / T chains per CTA, whole trajectories per
// launch.  TS >= T: threads' worth of shared memory per chain.  KM: evaluations
// per sweep between the first and the last of a trajectory (fewer in its last
// such sweep).
template <int TS, bool CUT, int KM, bool RAG, bool HF>
__global__ void __launch_bounds__(MARCH_CTA_THREADS, 2)
    march_lattice_kernel(const __grid_constant__ FusedArgs A, const __grid_constant__ Schedule S) {
    extern __shared__ float4 smem_f4[];
    const int T = A.march;
    const Geometry &g = A.g;
    for (int i = threadIdx.x; i < LOG1PEXP_NODES; i += blockDim.x) smem_f4[i] = A.lpe_tab[i];
    __syncthreads();
    const float4 *tab = smem_f4;
    const int group = threadIdx.x / T, groups = blockDim.x / T;
    const ChainThreads gr{(int)threadIdx.x - group * T, T, group + 1};
    const ChainThreads th = CUT ? ChainThreads{(int)threadIdx.x, (int)blockDim.x, 0} : gr;
    constexpr int FLOATS = march_floats(TS, KM, CUT) + MARCH_RED_BYTES / 4;
    float *smem = reinterpret_cast<float *>(smem_f4 + LOG1PEXP_NODES) + group * FLOATS;
    double *red = reinterpret_cast<double *>(
        reinterpret_cast<float *>(smem_f4 + LOG1PEXP_NODES) + (CUT ? 0 : group) * FLOATS + march_floats(TS, KM, CUT));
    int *bcast = reinterpret_cast<int *>(red + 8 * 8);
    double *const k0 = red + 8 * 8 + 1;   // the trajectory's K0

    const int chain = A.chain0 + (CUT ? (int)blockIdx.x : (int)blockIdx.x * groups + group);
    if (chain >= A.n_chains) return;   // (the other chains' barriers do not count these threads)
    // Little is kept in registers from pass to pass: a sweep of three
    // evaluations needs nearly all of them.
    ChainState *const st = A.state + chain;
    const ChainParams &prm = A.params[chain];
    const Cols cl = make_cols(g.X, gr.tid);
    MarchArgs M;
    M.z0 = CUT ? (int)((int64_t)group * g.nplanes / groups) : 0;
    M.nz = CUT ? (int)((int64_t)(group + 1) * g.nplanes / groups) - M.z0 : g.nplanes;
    M.ring = smem + 4 * gr.tid;
    M.edge = reinterpret_cast<float2 *>(smem + 2 * 4 * MARCH_SLOTS * TS);
    M.old_p = smem + (2 * 4 * MARCH_SLOTS + MARCH_SLOTS * KM * 4) * TS + 4 * gr.tid;
    const int64_t cbase = (int64_t)chain * g.N;
    M.p = A.p + cbase;
    int start = st->start;
    for (int k = 0; k < A.n_traj; ++k) {
        const uint32_t traj = A.traj0 + (uint32_t)k;
        M.traj = traj;
        // psi moves between the two buffers that do not hold the start
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
        // Evaluations j .. of a sweep.  Those between the first and the last go
        // KM = 3 to a sweep; what is left over joins the first evaluation's
        // sweep and, if need be, the last one's, so that no sweep of its own is
        // spent on it (the first and last sweeps are bound by arithmetic, not
        // by memory).  The sweep that also evaluates the start takes no guest.
        int j = 0;
        auto kk = [&](int i) { return kept((float)(S.kick[j + i] * prm.eps)); };
        auto dd = [&](int i) { return kept((float)(S.drift[j + i] * prm.eps)); };
        const int between = S.n_pass - 2;   // (n_pass >= 2)
        const bool ev_start = k == 0 && A.eval_start;
        const bool guest_first = !ev_start && between % KM >= 1;
        const bool guest_last = between % KM == 2 || (ev_start && between % KM == 1);
        {
            buffers();
            double v[1];
            if (ev_start) {
                Totals ini;
                const float kv[1] = {kk(0)}, dv[1] = {dd(0)};
                march_pass<TS, CUT, 1, true, false, true, RAG, HF>(A, M, gr, kv, dv, prm, cl, chain, tab, v, &ini);
                double ev[5] = {ini.S, ini.T, ini.AT, ini.HT, (double)ini.sS};
                chain_threads_sum<5>(ev, red, th);
                if (th.first()) {
                    st->S = ev[0];
                    set_obs(st, prm, ev[1], ev[2], ev[3], ev[4], 1.0 / (double)g.N);
                    st->prop = start;
                }
                j = 1;
            } else if (guest_first) {
                const float kv[2] = {kk(0), kk(1)}, dv[2] = {dd(0), dd(1)};
                march_pass<TS, CUT, 2, true, false, false, RAG, HF>(A, M, gr, kv, dv, prm, cl, chain, tab, v, nullptr);
                j = 2;
            } else {
                const float kv[1] = {kk(0)}, dv[1] = {dd(0)};
                march_pass<TS, CUT, 1, true, false, false, RAG, HF>(A, M, gr, kv, dv, prm, cl, chain, tab, v, nullptr);
                j = 1;
            }
            chain_threads_sum<1>(v, red, th);
            if (th.first()) *k0 = v[0];
            advance();
        }
        const int j_last = S.n_pass - 1 - (guest_last ? 1 : 0);   // the last sweep's first evaluation
        while (j < j_last) {
            buffers();
            if (j_last - j >= KM) {
                float kv[KM], dv[KM];
#pragma unroll
                for (int i = 0; i < KM; ++i) { kv[i] = kk(i); dv[i] = dd(i); }
                march_pass<TS, CUT, KM, false, false, false, RAG, HF>(A, M, gr, kv, dv, prm, cl, chain, tab, nullptr, nullptr);
                j += KM;
            } else {
                const float kv[1] = {kk(0)}, dv[1] = {dd(0)};
                march_pass<TS, CUT, 1, false, false, false, RAG, HF>(A, M, gr, kv, dv, prm, cl, chain, tab, nullptr, nullptr);
                j += 1;
            }
            advance();
        }
        buffers();
        Totals end;
        double K1;
        if (guest_last) {
            const float kv[2] = {kk(0), kk(1)}, dv[2] = {dd(0), 0.0f};
            march_pass<TS, CUT, 2, false, true, false, RAG, HF>(A, M, gr, kv, dv, prm, cl, chain, tab, &K1, &end);
            advance();
        } else {
            const float kv[1] = {kk(0)}, dv[1] = {0.0f};
            march_pass<TS, CUT, 1, false, true, false, RAG, HF>(A, M, gr, kv, dv, prm, cl, chain, tab, &K1, &end);
        }
        const int prop = src;   // the last evaluation itself writes no psi
        const double invN = 1.0 / (double)g.N;
        double w[6] = {K1, end.S, end.T, end.AT, end.HT, (double)end.sS};
        chain_threads_sum<6>(w, red, th);
        const double v[7] = {th.first() ? *k0 : 0.0, w[0], w[1], w[2], w[3], w[4], w[5]};
        double S_cur = th.first() ? st->S : 0.0;   // (kept by this thread alone)
        start = metropolis_step(th, A, st, prm, chain, traj, start, prop, v, invN, S_cur, true, bcast);
        if (A.flip_every > 0 && ((traj + 1) % (uint32_t)A.flip_every) == 0) {
            Acc fa = acc_zero();
            constexpr int SV = RAG ? 1 : 4;
            action_sweep<2, SV, false>(A, prm, chain, start, -1.0f, traj, A.seed,
                                       make_slots<SV>(g, gr.tid, gr.T), tab, fa, M.z0, M.z0 + M.nz);
            double wv[5] = {acc_val(fa.S, fa.Slo), kahan_val(fa.sT, fa.cT), kahan_val(fa.sAT, fa.cAT),
                            kahan_val(fa.sHT, fa.cHT), (double)fa.sS};
            chain_threads_sum<5>(wv, red, th);
            if (flip_step(th, A, st, prm, chain, traj, wv, invN, S_cur, true, bcast)) {
                const int f = (start != prop) ? 3 - start - prop : (start + 1) % 3;
                const float *gs = sel3(A, start) + cbase;
                float *gf = sel3(A, f) + cbase;
                for (int64_t i = th.tid; i < g.N; i += th.T) gf[i] = -gs[i];
                start = f;
                if (th.first()) st->start = f;
            }
            th.sync();
        }
        measure_step(th, A, st, traj, true);
    }
}

// How T-thread slabs fill CTAs of up to 256 threads (which share the 18 KB table
// of the action): several chains each as long as that leaves two CTAs for every
// SM; fewer chains than that are cut into slabs instead, as long as the slabs
// have rows enough (12 rows more than its own are computed per slab and sweep)
// and the SMs threads for them.  (Not for their shared memory: eight slabs of one warp take 117
// KB, each with a reduction block of which the chain uses one, so a single CTA of them
// fits on an SM and more chains than SMs take two turns.)  L = 251 x 173, 304 chains, minimum-norm integrator
// of 6 steps: 1.93 ms uncut (four warps per SM), 0.97 ms in four slabs; 64 chains
// of L = 128, N_md = 20: 0.18 ms in four slabs (1.53 ms on the plane-streaming
// kernel).
struct Packing {
    int per_cta, slabs;
};
inline Packing pack_chains(int n_chains, int T, int rows) {
    const int sms = sm_count();
    const int most = MARCH_CTA_THREADS / T;
    int n = most;
    while (n > 1 && (n_chains + n - 1) / n < 2 * sms) --n;
    if (n > 1) return {n, 1};
    int k = most;
    while (k > 1 && (rows / k < MARCH_MIN_SLAB || (int64_t)n_chains * T * k > 512 * (int64_t)sms)) --k;
    return {1, k};
}

template <int TS, bool CUT, bool RAG, bool HF>
cudaError_t node(const FusedArgs &a, int T, const Packing &pc, cudaKernelNodeParams *np, void **args) {
    auto kern = march_lattice_kernel<TS, CUT, MARCH_K, RAG, HF>;
    static DeviceOnce once;
    const cudaError_t e = allow_smem(once, kern, 227 * 1024);
    if (e != cudaSuccess) return e;
    const int n = a.n_chains - a.chain0, groups = pc.per_cta * pc.slabs;
    np->func = reinterpret_cast<void *>(kern);
    np->gridDim = dim3((unsigned)((n + pc.per_cta - 1) / pc.per_cta), 1, 1);
    np->blockDim = dim3((unsigned)(groups * T), 1, 1);
    np->sharedMemBytes = (unsigned)(LOG1PEXP_NODES * 16 +
                                    groups * (march_floats(TS, MARCH_K, CUT) * 4 + MARCH_RED_BYTES));
    np->kernelParams = args;
    np->extra = nullptr;
    return cudaSuccess;
}

template <bool RAG, bool HF>
cudaError_t node_ts(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args) {
    const Packing pc = pack_chains(a.n_chains - a.chain0, T, a.g.nplanes);
    if (pc.slabs > 1) {
        if (T <= 32) return node<32, true, RAG, HF>(a, T, pc, np, args);
        if (T <= 64) return node<64, true, RAG, HF>(a, T, pc, np, args);
        return node<128, true, RAG, HF>(a, T, pc, np, args);
    }
    if (T <= 32) return node<32, false, RAG, HF>(a, T, pc, np, args);
    if (T <= 64) return node<64, false, RAG, HF>(a, T, pc, np, args);
    if (T <= 128) return node<128, false, RAG, HF>(a, T, pc, np, args);
    return node<256, false, RAG, HF>(a, T, pc, np, args);
}

}  // namespace

// Kernel-node parameters of one kind of rows (one translation unit each,
// compiled in parallel): whole vectors or ragged, without or with a field.
cudaError_t march_node_vec(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args);
cudaError_t march_node_vec_field(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args);
cudaError_t march_node_rag(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args);
cudaError_t march_node_rag_field(const FusedArgs &a, int T, cudaKernelNodeParams *np, void **args);

}  // namespace ihmc
