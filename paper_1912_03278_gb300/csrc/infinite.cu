// infinite.cu -- FP32 HMC trajectories of the infinite-range (all-to-all)
// Ising model of the appendix, one CTA per chain, whole trajectories per
// launch.
//
// Connectivity K_ij = 1/N for i != j (0 on the diagonal), so with
// kappa = beta*J/N the matrix A = beta*J*K + C*1 acts as
//     (A x)_i = kappa * (sum_j x_j - x_i) + C * x_i :
// one block-wide sum per product and an O(N) per-site update, no GEMM.
// Per force evaluation (Sec. 3, F = A (tanh(A psi + h') - psi)):
//   sweep 1:  a = A psi,  t = tanh(a + h'),  u = t - psi,  U = sum_i u_i
//   sweep 2:  F = A u (from U),  p += kick*eps*F,  psi' = psi + drift*eps*p,
//             sum_i psi'_i for the next evaluation
// Each thread owns the same sites in both sweeps (site quads q = tid + k*nt).
// Two variants with bit-identical results:
//  * resident (N <= 32 * threads): the thread keeps its quads' psi, p and u in
//    registers for the whole trajectory; global memory is read once per
//    launch (and after a rejection) and written once per trajectory (the
//    proposal and the end momenta);
//  * streaming (any N): psi and p are re-read every pass, the leading quads'
//    from shared memory (struct Kept), the rest from global memory; sweep 2
//    recomputes u from psi with the identical instructions.
// Every sum adds the same per-quad partial sums in the same order in both,
// and the thread count depends on N alone.  The last pass of a trajectory also evaluates the
// proposal's action to FP64 accuracy in double-float arithmetic, the kinetic
// energies and the Sec. 4 estimators; the CTA takes the Metropolis decision
// itself (as the lattice kernel does).
//
// The updates and the action run on pairs of sites in packed FP32 instructions
// (pair.cuh: the scalar operations' bits): the resident kernel is bound by issue
// (2432 chains of N = 4096: 0.50 -> 0.47 ms per call of one trajectory), the streaming
// one by issue and latency (304 chains of N = 50001: 1.35 -> 1.14 ms; with kept
// quads 1.00, with batched loads 0.78).  128 registers at most (two CTAs of 256 threads on an SM);
// only the resident instances of eight quads a thread spill, 544 .. 648 bytes (stores).
#include <cuda_runtime.h>

#include "df32.cuh"
#include "device_common.cuh"
#include "internal.h"
#include "pair.cuh"

namespace ihmc {
namespace {

constexpr int INF_MAX_THREADS = 256;

// Four consecutive sites 4q..4q+3 of one chain; sites at or beyond N read as
// zero and are never stored.  V4: N is a multiple of 4, so a quad is one
// aligned float4.
struct Quad {
    pair_t a, b;   // held as pairs: the updates run on two sites per instruction
};
__device__ __forceinline__ Quad make_quad(float v0, float v1, float v2, float v3) {
    return Quad{pk(v0, v1), pk(v2, v3)};
}
__device__ __forceinline__ Quad make_quad(const float4 &t) { return make_quad(t.x, t.y, t.z, t.w); }
__device__ __forceinline__ void unpack(const Quad &q, float (&v)[4]) {
    upk(q.a, v[0], v[1]);
    upk(q.b, v[2], v[3]);
}
__device__ __forceinline__ float4 to_float4(const Quad &q) {
    float v[4];
    unpack(q, v);
    return make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ Quad quad_neg(const Quad &q) {
    const pair_t m = pk1(-1.0f);
    return Quad{mul2(q.a, m), mul2(q.b, m)};
}

template <bool V4>
__device__ __forceinline__ Quad ldq(const float *__restrict__ base, int64_t i0, int64_t N) {
    if constexpr (V4) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(base + i0);
        return Quad{t.x, t.y};
    } else {
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = (i0 + k < N) ? base[i0 + k] : 0.0f;
        return make_quad(v[0], v[1], v[2], v[3]);
    }
}

template <bool V4>
__device__ __forceinline__ void stq(float *__restrict__ base, int64_t i0, int64_t N, const Quad &r) {
    if constexpr (V4) {
        *reinterpret_cast<ulonglong2 *>(base + i0) = make_ulonglong2(r.a, r.b);
    } else {
        float v[4];
        unpack(r, v);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i0 + k < N) base[i0 + k] = v[k];
    }
}

// Number of valid sites in the quad starting at i0.
__device__ __forceinline__ int quad_len(int64_t i0, int64_t N) {
    const int64_t r = N - i0;
    return r >= 4 ? 4 : (int)r;
}

// Per-thread accumulators of one trajectory (same scheme as the lattice
// kernel: double-float energies with a separate low-word sum, Kahan FP32
// estimator sums).
struct Acc {
    f2 K0, K1, S;
    float K0lo, K1lo, Slo;
    float sT, cT, sAT, cAT, sHT, cHT;
    int sS;
};

__device__ __forceinline__ Acc acc_zero() {
    Acc a;
    a.K0 = a.K1 = a.S = f2{0.0f, 0.0f};
    a.K0lo = a.K1lo = a.Slo = 0.0f;
    a.sT = a.cT = a.sAT = a.cAT = a.sHT = a.cHT = 0.0f;
    a.sS = 0;
    return a;
}

// Per-chain constants: kappa = beta*J/N is stored in ChainParams::bJ.
struct InfConst {
    f2 C2, k2, hp2, beta2;
    float Cf, kf, betaf, hpf;
    bool hzero;
    const uint32_t *rk, *rk0;   // Philox key schedules of the seed and of key 0
};

__device__ __forceinline__ InfConst inf_const(const ChainParams &prm) {
    InfConst k;
    k.C2 = df_from_double(prm.C);
    k.k2 = df_from_double(prm.bJ);
    k.hp2 = df_from_double(prm.hp);
    k.beta2 = df_from_double(prm.beta);
    k.Cf = prm.Cf;
    k.kf = prm.bJf;
    k.betaf = prm.betaf;
    k.hpf = prm.hpf;
    k.hzero = prm.hp == 0.0;
    return k;
}

__device__ __forceinline__ float field_f(const FusedArgs &A, const InfConst &kc, int64_t i) {
    return A.hdf ? kc.betaf * A.hdf[i].x : kc.hpf;
}

// h' of the quad's sites.
__device__ __forceinline__ Quad quad_field(const FusedArgs &A, const InfConst &kc, int64_t i0, int n) {
    if (!A.hdf) return Quad{pk1(kc.hpf), pk1(kc.hpf)};
    float h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = (k < n) ? field_f(A, kc, i0 + k) : 0.0f;
    return make_quad(h[0], h[1], h[2], h[3]);
}

// t_i = tanh((A x)_i + h'_i) for the quad, with Sf = sum_j x_j in FP32: the
// one formula both the force sweeps and the estimators use.
__device__ __forceinline__ Quad quad_tanh(const FusedArgs &A, const InfConst &kc, const Quad &x,
                                          float Sf, int64_t i0, int n) {
    const Quad h = quad_field(A, kc, i0, n);
    const pair_t C = pk1(kc.Cf), k = pk1(kc.kf), S = pk1(Sf);
    return Quad{tanh2(add2(fma2(C, x.a, mul2(k, sub2(S, x.a))), h.a)),
                tanh2(add2(fma2(C, x.b, mul2(k, sub2(S, x.b))), h.b))};
}

// Action terms of the quad's sites of S(x) (Sec. 2, Eq. phi_psi_substitution:
// S_i = 1/2 x_i a_i - |y_i| - log(1 + exp(-2|y_i|)), a = A x, y = a + h') in
// double-float arithmetic with Sx = sum_j x_j as a double-float; the Sec. 4
// estimator sums from the force-form tanh values t, and one conditional spin
// draw per site.
__device__ __forceinline__ void quad_action(const FusedArgs &A, const InfConst &kc, const Quad &x,
                                            const Quad &t, f2 Sx, int64_t i0, int n,
                                            uint32_t spin_traj, const uint32_t *seed, int chain,
                                            const float4 *tab, Acc &acc) {
    const float4 w = spin_u4((uint32_t)(i0 >> 2), spin_traj, (uint32_t)chain, seed);
    const float su[4] = {w.x, w.y, w.z, w.w};
    const bool has_h = A.hdf || !kc.hzero;
    f2 si[4];
    float ahi[4], tv[4], hf[4];
    unpack(t, tv);
    unpack(quad_field(A, kc, i0, n), hf);
#pragma unroll
    for (int q = 0; q < 2; ++q) {   // sites beyond n are computed and left out below
        const pair_t ps = q ? x.b : x.a;
        // sum over j != i
        const f2x2 off = df_add_f(f2x2{pk1(Sx.hi), pk1(Sx.lo)}, mul2(ps, pk1(-1.0f)));
        const f2x2 C2 = dup_df(kc.C2), k2 = dup_df(kc.k2);
        const f2x2 a = df_add_q(df_mul_fc(C2, pk1(-kc.C2.hi), ps), df_mul(k2, pk1(-kc.k2.hi), off));
        f2x2 y = a;
        if (A.hdf) {
            f2 h0{0.0f, 0.0f}, h1{0.0f, 0.0f};
            if (2 * q < n) {
                const float2 hh = A.hdf[i0 + 2 * q];
                h0 = df_mul(kc.beta2, f2{hh.x, hh.y});
            }
            if (2 * q + 1 < n) {
                const float2 hh = A.hdf[i0 + 2 * q + 1];
                h1 = df_mul(kc.beta2, f2{hh.x, hh.y});
            }
            y = df_add_q(a, f2x2{pk(h0.hi, h1.hi), pk(h0.lo, h1.lo)});
        } else if (!kc.hzero) {
            y = df_add_q(a, dup_df(kc.hp2));
        }
        upk(action_term(ps, a, y, tab), si[2 * q], si[2 * q + 1]);
        upk(a.hi, ahi[2 * q], ahi[2 * q + 1]);
    }
    f2 sv{0.0f, 0.0f};
    float vT = 0.0f, vAT = 0.0f, vHT = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k >= n) break;
        sv = k ? df_add_q(sv, si[k]) : si[k];
        vT += tv[k];
        vAT = fmaf(ahi[k], tv[k], vAT);
        if (has_h) vHT = fmaf(hf[k], tv[k], vHT);
        acc.sS += (su[k] < (1.0f + tv[k]) * 0.5f) ? 1 : -1;
    }
    acc_add(acc.S, acc.Slo, sv);
    kahan_add(acc.sT, acc.cT, vT);
    kahan_add(acc.sAT, acc.cAT, vAT);
    if (has_h) kahan_add(acc.sHT, acc.cHT, vHT);
}

__device__ __forceinline__ float *sel3(const FusedArgs &A, int i) {
    return i == 0 ? A.psi[0] : (i == 1 ? A.psi[1] : A.psi[2]);
}

// Sum of the quad's valid sites.  Every sum over a configuration adds these
// quad sums in the same order (thread t: quads t, t + nt, ...; then the block
// sum), so the sum kept while drifting equals the one recomputed from the
// stored buffer bit for bit, and the force stays a function of psi alone.
__device__ __forceinline__ float quad_sum(const Quad &q, int n) {
    float v[4];
    unpack(q, v);
    const float a = v[0] + (n > 1 ? v[1] : 0.0f);
    const float b = (n > 2 ? v[2] : 0.0f) + (n > 3 ? v[3] : 0.0f);
    return a + b;
}

// Kinetic energy of the quad's first n sites, added site by site.
__device__ __forceinline__ void quad_kinetic(const Quad &p, int n, f2 &K, float &Klo) {
    f2 v[4];
    upk(half_square(p.a), v[0], v[1]);
    upk(half_square(p.b), v[2], v[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < n) acc_add(K, Klo, v[k]);
}

// p += kick F with F = A u, and x + drift p.
__device__ __forceinline__ Quad quad_kick(const InfConst &kc, float kick, const Quad &p, const Quad &u, float Uf) {
    const pair_t C = pk1(kc.Cf), k = pk1(kc.kf), U = pk1(Uf), e = pk1(kick);
    return Quad{fma2(e, fma2(C, u.a, mul2(k, sub2(U, u.a))), p.a),
                fma2(e, fma2(C, u.b, mul2(k, sub2(U, u.b))), p.b)};
}
__device__ __forceinline__ Quad quad_axpy(float d, const Quad &p, const Quad &x) {
    const pair_t e = pk1(d);
    return Quad{fma2(e, p.a, x.a), fma2(e, p.b, x.b)};
}
__device__ __forceinline__ Quad quad_sub(const Quad &a, const Quad &b) { return Quad{sub2(a.a, b.a), sub2(a.b, b.b)}; }

// CTA-wide sums in FP32-pipe arithmetic (FP64 issues at a small fraction of
// the FP32 rate on GB300), blockDim a multiple of 32 and at most 256.  The
// order is fixed and the same in every thread: a shuffle tree to lane 0 of
// each warp, then lanes 0..7 of every warp over the per-warp totals.
struct Red {
    float *f;   // 2 x 8 floats, halves used alternately: one barrier per sum
    f2 *d;      // 8 x 8 double-floats
    int par;
};

__device__ __forceinline__ float bsum_f32(float v, Red &r) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    float *buf = r.f + 8 * r.par;
    r.par ^= 1;
    if (lane == 0) buf[warp] = v;
    __syncthreads();
    float w = lane < (int)(blockDim.x >> 5) ? buf[lane] : 0.0f;
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) w += __shfl_down_sync(0xffffffffu, w, off);
    return __shfl_sync(0xffffffffu, w, 0);
}

__device__ __forceinline__ f2 shfl_down_f2(f2 v, int off) {
    return f2{__shfl_down_sync(0xffffffffu, v.hi, off), __shfl_down_sync(0xffffffffu, v.lo, off)};
}

template <int NV>
__device__ __forceinline__ void bsum_f2(f2 (&v)[NV], Red &r) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[k] = df_add(v[k], shfl_down_f2(v[k], off));
    __syncthreads();   // earlier readers of r.d are done
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) r.d[warp * NV + k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        f2 w = lane < (int)(blockDim.x >> 5) ? r.d[lane * NV + k] : f2{0.0f, 0.0f};
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) w = df_add(w, shfl_down_f2(w, off));
        v[k] = f2{__shfl_sync(0xffffffffu, w.hi, 0), __shfl_sync(0xffffffffu, w.lo, 0)};
    }
}

// Sum of a configuration: the thread's partial over its quads (double-float,
// quads in increasing order) and the FP32 CTA total of the partials' high
// words, the value the force uses.  The double-float CTA total (the action's
// value) is formed from the partials only where the action needs it.
// Negation is exact in every step, so the sum of -psi is the negated sum.
struct CSum {
    f2 part;
    float Sf;
};

__device__ __forceinline__ CSum csum_make(f2 part, Red &r) { return CSum{part, bsum_f32(part.hi, r)}; }
__device__ __forceinline__ CSum csum_neg(const CSum &c) { return CSum{df_neg(c.part), -c.Sf}; }
__device__ __forceinline__ f2 csum_exact(const CSum &c, Red &r) {
    f2 v[1] = {c.part};
    bsum_f2<1>(v, r);
    return v[0];
}

// Sum of one chain's buffer.
template <bool V4>
__device__ CSum chain_sum(const float *__restrict__ x, int64_t N, Red &r) {
    const int64_t nq = (N + 3) >> 2;
    f2 s{0.0f, 0.0f};
    for (int64_t q = threadIdx.x; q < nq; q += blockDim.x) {
        const int64_t i0 = 4 * q;
        s = df_add_f(s, quad_sum(ldq<V4>(x, i0, N), quad_len(i0, N)));
    }
    return csum_make(s, r);
}

struct PassCfg {
    int src, dst;
    float kick, drift;   // already multiplied by eps
    uint32_t traj;
};

// The streaming variant's quads that stay in shared memory through a
// trajectory: psi of the thread's first nx quads, p of its first np, slot
// k * nt + tid each (written and read by the owning thread only).  What bounds the
// variant besides issue is the L2: every evaluation moves 20 B per site through
// it, and two psi buffers and p of 304 chains of N = 50000 (183 MB) do not fit
// into its 129 MB.  psi is kept before p (three of the five accesses against two), and the
// passes after the first drift in place, which leaves one psi buffer in use.
// Kernel, one trajectory of N_md = 10, ms: 304 chains of N = 50000 0.92 -> 0.64,
// 50001 0.97 -> 0.85, 20000 0.225 -> 0.195.
struct Kept {
    ulonglong2 *x, *p;
    int nx, np;
};
__device__ __forceinline__ Quad lds_quad(const ulonglong2 &v) { return Quad{v.x, v.y}; }

// A quad inside the chain, without bounds checks.
template <bool V4>
__device__ __forceinline__ Quad ldq4(const float *p) {
    if constexpr (V4) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
        return Quad{t.x, t.y};
    } else {
        return make_quad(p[0], p[1], p[2], p[3]);
    }
}
template <bool V4>
__device__ __forceinline__ void stq4(float *p, const Quad &r) {
    if constexpr (V4) {
        *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(r.a, r.b);
    } else {
        float v[4];
        unpack(r, v);
#pragma unroll
        for (int k = 0; k < 4; ++k) p[k] = v[k];
    }
}

// Quads per thread whose loads the middle passes issue together.  With 16 warps
// on an SM the latency of the L2 bounded them (long-scoreboard stalls 1.36 per
// issue at N = 20001), and the bounds checks of every quad kept loads from
// being issued ahead.  One trajectory of N_md = 10, ms, without / 1 / 2 / 4 in a batch:
// 304 chains of N = 50001 0.85 / 0.73 / 0.65 / 0.63, 50000 0.62 / 0.60 / 0.60 / 0.51, 20001
// 0.250 / 0.234 / 0.219 / 0.225, 9000 0.102 / 0.100 / 0.100 / 0.097; 608 of 65536 1.84 / 1.75 / 1.74 /
// 1.42; 152 of 200000 2.86 / 2.56 / 2.54 / 1.81.
constexpr int INF_BATCH = 4;

// One force evaluation.  cs: sum of the source configuration on entry, of
// the drifted one on exit (unchanged by the last pass, which does not drift).
// The first pass drifts from the current configuration into the proposal's
// buffer, the later ones in place (src == dst: a thread overwrites only the
// quad it has just read); kept quads reach the buffers in the last pass.
template <bool V4, bool FIRST, bool LAST>
__device__ void inf_pass(const FusedArgs &A, const PassCfg &pc, const InfConst &kc, int chain,
                         const Kept &kp, CSum &cs, Red &red, const float4 *tab, Acc &acc) {
    const int64_t N = A.g.N;
    const int64_t nq = (N + 3) >> 2;
    const int64_t cbase = (int64_t)chain * N;
    const float *src = sel3(A, pc.src) + cbase;
    float *dst = sel3(A, pc.dst) + cbase;
    float *gp = A.p + cbase;
    const float Sf = cs.Sf;

    // ---- sweep 1: U = sum_i (tanh(A psi + h')_i - psi_i) ----
    float su = 0.0f;
    f2 Sdf{0.0f, 0.0f};
    if constexpr (LAST) Sdf = csum_exact(cs, red);
    constexpr int NT = INF_MAX_THREADS;   // the block size of every chain that streams
    // rows of whole quads, for which the middle passes need no bounds
    const int rows = (FIRST || LAST) ? 0 : (int)(N / (4 * NT)) / INF_BATCH * INF_BATCH;
    int k = 0;
    for (; k < rows; k += INF_BATCH) {
        const int64_t q = threadIdx.x + (int64_t)k * NT;
        Quad x[INF_BATCH];
#pragma unroll
        for (int b = 0; b < INF_BATCH; ++b)
            x[b] = k + b < kp.nx ? lds_quad(kp.x[q + b * NT]) : ldq4<V4>(src + 4 * (q + b * NT));
#pragma unroll
        for (int b = 0; b < INF_BATCH; ++b)
            su += quad_sum(quad_sub(quad_tanh(A, kc, x[b], Sf, 4 * (q + b * NT), 4), x[b]), 4);
    }
    for (int64_t q = threadIdx.x + (int64_t)k * NT; q < nq; q += NT, ++k) {
        const int64_t i0 = 4 * q;
        const int n = quad_len(i0, N);
        Quad x;
        if (!FIRST && k < kp.nx) {
            x = lds_quad(kp.x[q]);
            if constexpr (LAST) stq<V4>(dst, i0, N, x);
        } else {
            x = ldq<V4>(src, i0, N);
            if (FIRST && k < kp.nx) kp.x[q] = make_ulonglong2(x.a, x.b);
        }
        const Quad t = quad_tanh(A, kc, x, Sf, i0, n);
        su += quad_sum(quad_sub(t, x), n);
        // the last pass's configuration is the proposal
        if constexpr (LAST) quad_action(A, kc, x, t, Sdf, i0, n, pc.traj, kc.rk, chain, tab, acc);
    }
    const float Uf = bsum_f32(su, red);

    // ---- sweep 2: kick with F = A u, drift ----
    f2 sp{0.0f, 0.0f};
    k = 0;
    for (; k < rows; k += INF_BATCH) {
        const int64_t q = threadIdx.x + (int64_t)k * NT;
        Quad x[INF_BATCH], pv[INF_BATCH];
#pragma unroll
        for (int b = 0; b < INF_BATCH; ++b) {
            x[b] = k + b < kp.nx ? lds_quad(kp.x[q + b * NT]) : ldq4<V4>(src + 4 * (q + b * NT));
            pv[b] = k + b < kp.np ? lds_quad(kp.p[q + b * NT]) : ldq4<V4>(gp + 4 * (q + b * NT));
        }
#pragma unroll
        for (int b = 0; b < INF_BATCH; ++b) {
            const Quad t = quad_tanh(A, kc, x[b], Sf, 4 * (q + b * NT), 4);
            pv[b] = quad_kick(kc, pc.kick, pv[b], quad_sub(t, x[b]), Uf);
            x[b] = quad_axpy(pc.drift, pv[b], x[b]);
            sp = df_add_f(sp, quad_sum(x[b], 4));
            if (k + b < kp.np) kp.p[q + b * NT] = make_ulonglong2(pv[b].a, pv[b].b);
            else stq4<V4>(gp + 4 * (q + b * NT), pv[b]);
            if (k + b < kp.nx) kp.x[q + b * NT] = make_ulonglong2(x[b].a, x[b].b);
            else stq4<V4>(dst + 4 * (q + b * NT), x[b]);
        }
    }
    for (int64_t q = threadIdx.x + (int64_t)k * NT; q < nq; q += NT, ++k) {
        const int64_t i0 = 4 * q;
        const int n = quad_len(i0, N);
        Quad x, pv;
        if (k < kp.nx) x = lds_quad(kp.x[q]);
        else x = ldq<V4>(src, i0, N);
        if constexpr (FIRST) {
            pv = make_quad(momenta4((uint32_t)q, pc.traj, (uint32_t)chain, kc.rk));
            quad_kinetic(pv, n, acc.K0, acc.K0lo);
        } else if (k < kp.np) {
            pv = lds_quad(kp.p[q]);
        } else {
            pv = ldq<V4>(gp, i0, N);
        }
        const Quad t = quad_tanh(A, kc, x, Sf, i0, n);
        pv = quad_kick(kc, pc.kick, pv, quad_sub(t, x), Uf);
        if (!LAST && k < kp.np) kp.p[q] = make_ulonglong2(pv.a, pv.b);
        else stq<V4>(gp, i0, N, pv);
        if constexpr (LAST) {
            quad_kinetic(pv, n, acc.K1, acc.K1lo);
        } else {
            const Quad xn = quad_axpy(pc.drift, pv, x);
            if (k < kp.nx) kp.x[q] = make_ulonglong2(xn.a, xn.b);
            else stq<V4>(dst, i0, N, xn);
            sp = df_add_f(sp, quad_sum(xn, n));
        }
    }
    if constexpr (!LAST) cs = csum_make(sp, red);
}

// Action S(sign*x) of the chain's buffer `buf` with the estimators and one
// conditional spin draw per site (evaluation of the current state, sign
// flip proposal).
template <bool V4>
__device__ void inf_action(const FusedArgs &A, const InfConst &kc, int chain, int buf, float sign,
                           uint32_t spin_traj, const uint32_t *seed, Red &red, const float4 *tab,
                           Acc &acc) {
    const int64_t N = A.g.N;
    const int64_t nq = (N + 3) >> 2;
    const float *__restrict__ x = sel3(A, buf) + (int64_t)chain * N;
    CSum c = chain_sum<V4>(x, N, red);
    if (sign < 0.0f) c = csum_neg(c);
    const float Sf = c.Sf;
    const f2 Sdf = csum_exact(c, red);
    for (int64_t q = threadIdx.x; q < nq; q += blockDim.x) {
        const int64_t i0 = 4 * q;
        const int n = quad_len(i0, N);
        Quad v = ldq<V4>(x, i0, N);
        if (sign < 0.0f) v = quad_neg(v);
        const Quad t = quad_tanh(A, kc, v, Sf, i0, n);
        quad_action(A, kc, v, t, Sdf, i0, n, spin_traj, seed, chain, tab, acc);
    }
}

__device__ __forceinline__ int buf_loc(int start, int j) {
    if (j == 0) return start;
    return (start + ((j & 1) ? 1 : 2)) % 3;
}

__device__ __forceinline__ void set_obs(ChainState *st, const ChainParams &prm, double sT,
                                        double sAT, double sHT, double sS, double invN) {
    const double m = sT * invN;
    st->obs[0] = m;
    st->obs[1] = 0.5 * prm.C - 0.5 * sAT * invN - sHT * invN;
    st->obs[2] = fabs(sS) * invN;
    st->obs[3] = fabs(m);
}

// Metropolis decision of trajectory traj (Sec. 3) from the block totals v =
// {K0, K1, S1, sum t, sum a.t, sum h'.t, sum of spins} of the proposal held
// in buffer prop; thread 0 updates the chain state.  Returns the buffer of
// the chain's current configuration afterwards (in every thread).
__device__ int metropolis(const FusedArgs &A, ChainState *st, const ChainParams &prm, int chain,
                          uint32_t traj, int start, int prop, const double (&v)[7], double invN,
                          int *bcast) {
    if (threadIdx.x == 0) {
        const double S0 = st->S;
        const double dH = (v[1] + v[2]) - (v[0] + S0);
        const double logu = accept_logu(traj, (uint32_t)chain, A.seed, PURPOSE_ACC);
        const bool accd = logu < -dH;
        st->prop = prop;
        st->rec[ISING_REC_DH] = dH;
        st->rec[ISING_REC_LOGU] = logu;
        st->rec[ISING_REC_ACCEPTED] = accd ? 1.0 : 0.0;
        st->rec[ISING_REC_K0] = v[0];
        st->rec[ISING_REC_S0] = S0;
        st->rec[ISING_REC_K1] = v[1];
        st->rec[ISING_REC_S1] = v[2];
        st->rec[ISING_REC_FLIPPED] = 0.0;
        if (accd) {
            st->start = prop;
            st->S = v[2];
            set_obs(st, prm, v[3], v[4], v[5], v[6], invN);
        }
        bcast[0] = accd ? prop : start;
    }
    __syncthreads();
    const int cur = bcast[0];
    __syncthreads();
    return cur;
}

// Sign-flip proposal psi -> -psi (Sec. 3) from the block totals w = {S(-psi),
// sum t, sum a.t, sum h'.t, sum of spins}; returns 1 (every thread) if taken.
__device__ int flip_decision(const FusedArgs &A, ChainState *st, const ChainParams &prm, int chain,
                             uint32_t traj, const double (&w)[5], double invN, int *bcast) {
    if (threadIdx.x == 0) {
        const double lu = accept_logu(traj, (uint32_t)chain, A.seed, PURPOSE_FLIP);
        const bool fl = lu < -(w[0] - st->S);
        if (fl) {
            st->S = w[0];
            set_obs(st, prm, w[1], w[2], w[3], w[4], invN);
            st->rec[ISING_REC_FLIPPED] = 1.0;
        }
        bcast[1] = fl ? 1 : 0;
    }
    __syncthreads();
    const int fl = bcast[1];
    __syncthreads();
    return fl;
}

// Measurement after the Metropolis step: a repeated configuration repeats its
// measurement (thread 0).
__device__ __forceinline__ void measure(const FusedArgs &A, ChainState *st, uint32_t traj) {
    if (threadIdx.x == 0 && (int64_t)traj >= (int64_t)A.n_therm) {
        double *sm = st->sums;
        const double dH = st->rec[ISING_REC_DH];
        sm[ISING_SUM_NMEAS] += 1.0;
        sm[ISING_SUM_NACC] += st->rec[ISING_REC_ACCEPTED];
        sm[ISING_SUM_M] += st->obs[0];
        sm[ISING_SUM_M2] += st->obs[0] * st->obs[0];
        sm[ISING_SUM_E] += st->obs[1];
        sm[ISING_SUM_E2] += st->obs[1] * st->obs[1];
        sm[ISING_SUM_ABSM] += st->obs[2];
        sm[ISING_SUM_ABSM2] += st->obs[2] * st->obs[2];
        sm[ISING_SUM_DH] += dH;
        sm[ISING_SUM_EXPMDH] += exp(-dH);
    }
    __syncthreads();
}

// CTA totals of a trajectory's accumulators as doubles, identical in every
// thread: {K0, K1, S, sum t, sum a.t, sum h'.t, sum of spins}.  The
// per-thread values enter as exact double-floats.
__device__ __forceinline__ f2 int_f2(int n) {
    const float hi = (float)n;
    return f2{hi, (float)(n - (int)hi)};
}

__device__ __forceinline__ void acc_totals(const Acc &acc, double (&v)[7], Red &red) {
    f2 t[7] = {df_add_f(acc.K0, acc.K0lo), df_add_f(acc.K1, acc.K1lo), df_add_f(acc.S, acc.Slo),
               two_sum(acc.sT, -acc.cT),  two_sum(acc.sAT, -acc.cAT), two_sum(acc.sHT, -acc.cHT),
               int_f2(acc.sS)};
    bsum_f2<7>(t, red);
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = df_to_double(t[k]);
}

// The same for an action sweep: {S, sum t, sum a.t, sum h'.t, sum of spins}.
__device__ __forceinline__ void action_totals(const Acc &acc, double (&w)[5], Red &red) {
    f2 t[5] = {df_add_f(acc.S, acc.Slo), two_sum(acc.sT, -acc.cT), two_sum(acc.sAT, -acc.cAT),
               two_sum(acc.sHT, -acc.cHT), int_f2(acc.sS)};
    bsum_f2<5>(t, red);
#pragma unroll
    for (int k = 0; k < 5; ++k) w[k] = df_to_double(t[k]);
}

// ---------------------------------------------------------------- resident --
// The thread's quads q = tid + k*nt, k < QPT, held in registers: x (psi), pm
// (p); u between the two sweeps in shared memory (us[q], written and read by
// the owning thread only).  One force evaluation, the same arithmetic in the
// same order as inf_pass.  The first pass's momentum draw and the last pass's
// action run in loops that are not unrolled, through a second shared array
// (aux[q], again the owning thread's only): their code then appears once, not
// once per quad, which keeps the kernel's instruction footprint small.
template <bool V4, int QPT, bool FULL, bool FIRST, bool LAST>
__device__ __forceinline__ void res_pass(const FusedArgs &A, const InfConst &kc, int chain,
                                         uint32_t traj, float kick, float drift, Quad (&x)[QPT],
                                         Quad (&pm)[QPT], float4 *us, CSum &cs, Red &red,
                                         const float4 *tab, Acc &acc) {
    const int64_t N = A.g.N;
    const int64_t nq = (N + 3) >> 2;
    const float Sf = cs.Sf;
    float4 *aux = us + QPT * blockDim.x;
    constexpr bool ONE_PASS = FIRST && LAST;   // (never with two or more passes)
    if constexpr (FIRST && !ONE_PASS) {
#pragma unroll 1
        for (int k = 0; k < QPT; ++k) {
            const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
            if (FULL || q < nq) aux[q] = momenta4((uint32_t)q, traj, (uint32_t)chain, kc.rk);
        }
    }
    float su = 0.0f;
    f2 Sdf{0.0f, 0.0f};
    if constexpr (LAST) Sdf = csum_exact(cs, red);
#pragma unroll
    for (int k = 0; k < QPT; ++k) {
        const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
        if (FULL || q < nq) {
            const int64_t i0 = 4 * q;
            const int n = (FULL ? 4 : quad_len(i0, N));
            const Quad t = quad_tanh(A, kc, x[k], Sf, i0, n);
            const Quad u = quad_sub(t, x[k]);
            us[q] = to_float4(u);
            su += quad_sum(u, n);
            if constexpr (ONE_PASS)
                quad_action(A, kc, x[k], t, Sdf, i0, n, traj, kc.rk, chain, tab, acc);
            else if constexpr (LAST)
                aux[q] = to_float4(x[k]);
        }
    }
    if constexpr (LAST && !ONE_PASS) {
        // the proposal's action, quads in the same order (t recomputed: the
        // same function of the same values)
#pragma unroll 1
        for (int k = 0; k < QPT; ++k) {
            const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
            if (FULL || q < nq) {
                const int64_t i0 = 4 * q;
                const int n = (FULL ? 4 : quad_len(i0, N));
                const Quad xq = make_quad(aux[q]);
                const Quad t = quad_tanh(A, kc, xq, Sf, i0, n);
                quad_action(A, kc, xq, t, Sdf, i0, n, traj, kc.rk, chain, tab, acc);
            }
        }
    }
    const float Uf = bsum_f32(su, red);
    f2 sp{0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < QPT; ++k) {
        const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
        if (FULL || q < nq) {
            const int n = (FULL ? 4 : quad_len(4 * q, N));
            if constexpr (FIRST) {
                pm[k] = make_quad(ONE_PASS ? momenta4((uint32_t)q, traj, (uint32_t)chain, kc.rk) : aux[q]);
                quad_kinetic(pm[k], n, acc.K0, acc.K0lo);
            }
            pm[k] = quad_kick(kc, kick, pm[k], make_quad(us[q]), Uf);
            if constexpr (LAST) {
                quad_kinetic(pm[k], n, acc.K1, acc.K1lo);
            } else {
                x[k] = quad_axpy(drift, pm[k], x[k]);
                sp = df_add_f(sp, quad_sum(x[k], n));
            }
        }
    }
    if constexpr (!LAST) cs = csum_make(sp, red);
}

template <bool V4, int QPT, bool FULL>
__device__ __forceinline__ void res_load(const float *__restrict__ g, int64_t N, Quad (&x)[QPT]) {
    const int64_t nq = (N + 3) >> 2;
#pragma unroll
    for (int k = 0; k < QPT; ++k) {
        const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
        if (FULL || q < nq) x[k] = ldq<V4>(g, 4 * q, N);
    }
}

template <bool V4, int QPT, bool FULL>
__device__ __forceinline__ void res_store(float *__restrict__ g, int64_t N, const Quad (&x)[QPT]) {
    const int64_t nq = (N + 3) >> 2;
#pragma unroll
    for (int k = 0; k < QPT; ++k) {
        const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
        if (FULL || q < nq) stq<V4>(g, 4 * q, N, x[k]);
    }
}

// Whole trajectories with the chain resident in registers.  Every thread
// reads and writes only its own quads, so no barrier guards global memory.
template <bool V4, int QPT, bool FULL>
__device__ void res_trajectories(const FusedArgs &A, const Schedule &S, const ChainParams &prm,
                                 const InfConst &kc, ChainState *st, int chain, double invN,
                                 float4 *us, Red &red, int *bcast, const float4 *tab) {
    const int64_t N = A.g.N;
    const int64_t nq = (N + 3) >> 2;
    const int64_t cbase = (int64_t)chain * N;
    Quad x[QPT], pm[QPT];
#pragma unroll
    for (int k = 0; k < QPT; ++k) x[k] = pm[k] = Quad{0ull, 0ull};
    int start = st->start;
    res_load<V4, QPT, FULL>(sel3(A, start) + cbase, N, x);
    // sum of the current configuration (the order of chain_sum)
    CSum Sstart;
    {
        f2 s{0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < QPT; ++k) {
            const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
            if (FULL || q < nq) s = df_add_f(s, quad_sum(x[k], (FULL ? 4 : quad_len(4 * q, N))));
        }
        Sstart = csum_make(s, red);
    }
    for (int it = 0; it < A.n_traj; ++it) {
        const uint32_t traj = A.traj0 + (uint32_t)it;
        Acc acc = acc_zero();
        CSum cs = Sstart;
        for (int j = 0; j < S.n_pass; ++j) {
            const float kick = (float)(S.kick[j] * prm.eps);
            const float drift = (float)(S.drift[j] * prm.eps);
            const bool first = j == 0, last = j == S.n_pass - 1;
            if (first && last)
                res_pass<V4, QPT, FULL, true, true>(A, kc, chain, traj, kick, drift, x, pm, us, cs, red, tab, acc);
            else if (first)
                res_pass<V4, QPT, FULL, true, false>(A, kc, chain, traj, kick, drift, x, pm, us, cs, red, tab, acc);
            else if (last)
                res_pass<V4, QPT, FULL, false, true>(A, kc, chain, traj, kick, drift, x, pm, us, cs, red, tab, acc);
            else
                res_pass<V4, QPT, FULL, false, false>(A, kc, chain, traj, kick, drift, x, pm, us, cs, red, tab, acc);
        }
        // the proposal and the end momenta go to global memory
        const int prop = buf_loc(start, S.n_pass - 1);
        res_store<V4, QPT, FULL>(sel3(A, prop) + cbase, N, x);
        res_store<V4, QPT, FULL>(A.p + cbase, N, pm);
        double v[7];
        acc_totals(acc, v, red);
        const int cur = metropolis(A, st, prm, chain, traj, start, prop, v, invN, bcast);
        if (cur == start) res_load<V4, QPT, FULL>(sel3(A, start) + cbase, N, x);   // rejected
        else Sstart = cs;                                                   // the proposal's sum
        start = cur;
        if (A.flip_every > 0 && ((traj + 1) % (uint32_t)A.flip_every) == 0) {
            // action of -psi from the registers (the arithmetic of inf_action)
            Acc fa = acc_zero();
            const CSum neg = csum_neg(Sstart);
            const float Sf = neg.Sf;
            const f2 Sdf = csum_exact(neg, red);
#pragma unroll
            for (int k = 0; k < QPT; ++k) {
                const int64_t q = threadIdx.x + (int64_t)k * blockDim.x;
                if (FULL || q < nq) {
                    const int64_t i0 = 4 * q;
                    const int n = (FULL ? 4 : quad_len(i0, N));
                    const Quad v4 = quad_neg(x[k]);
                    const Quad t = quad_tanh(A, kc, v4, Sf, i0, n);
                    quad_action(A, kc, v4, t, Sdf, i0, n, traj, kc.rk, chain, tab, fa);
                }
            }
            double w[5];
            action_totals(fa, w, red);
            if (flip_decision(A, st, prm, chain, traj, w, invN, bcast)) {
                const int f = (start != prop) ? 3 - start - prop : (start + 1) % 3;
#pragma unroll
                for (int k = 0; k < QPT; ++k) x[k] = quad_neg(x[k]);
                res_store<V4, QPT, FULL>(sel3(A, f) + cbase, N, x);
                start = f;
                Sstart = neg;
                if (threadIdx.x == 0) st->start = f;
            }
        }
        measure(A, st, traj);
    }
}

// QPT > 0: the resident variant with QPT quads per thread (trajectories
// only); QPT = 0: streaming.  FULL (resident, N a multiple of 4 and every
// thread's QPT quads inside the chain): the bounds and quad-length checks
// fold away; the arithmetic and its order are those of the general instance.
template <bool V4, int QPT, bool FULL = false>
__global__ void __launch_bounds__(INF_MAX_THREADS, 2)
    infinite_kernel(const __grid_constant__ FusedArgs A, const __grid_constant__ Schedule S) {
    __shared__ float4 tab_s[LOG1PEXP_NODES];
    __shared__ float red_f[16];
    __shared__ f2 red_d[64];
    __shared__ int bcast[2];
    extern __shared__ float4 us[];   // resident variant: u and aux, QPT * blockDim.x quads each
    const int chain = A.chain0 + blockIdx.x;
    if (chain >= A.n_chains) return;
    const int64_t N = A.g.N;
    ChainState *st = A.state + chain;
    const ChainParams prm = A.params[chain];
    const double invN = 1.0 / (double)N;

    if (A.mode == MODE_MOMENTA) {
        float *gp = A.p + (int64_t)chain * N;
        for (int64_t q = threadIdx.x; q < ((N + 3) >> 2); q += blockDim.x) {
            stq<V4>(gp, 4 * q, N, make_quad(momenta4((uint32_t)q, A.traj0, (uint32_t)chain, A.round_keys)));
        }
        return;
    }
    for (int i = threadIdx.x; i < LOG1PEXP_NODES; i += blockDim.x) tab_s[i] = A.lpe_tab[i];
    __syncthreads();
    InfConst kc = inf_const(prm);
    kc.rk = A.round_keys;
    kc.rk0 = A.round_keys0;
    Red red{red_f, red_d, 0};

    if (A.mode == MODE_EVAL) {
        Acc acc = acc_zero();
        const int start = st->start;
        inf_action<V4>(A, kc, chain, start, 1.0f, TRAJ_INIT, kc.rk0, red, tab_s, acc);
        double v[5];
        action_totals(acc, v, red);
        if (threadIdx.x == 0) {
            st->S = v[0];
            set_obs(st, prm, v[1], v[2], v[3], v[4], invN);
            st->prop = start;
        }
        return;
    }
    if constexpr (QPT > 0) {
        res_trajectories<V4, QPT, FULL>(A, S, prm, kc, st, chain, invN, us, red, bcast, tab_s);
        return;
    }

    Kept kp;
    {
        uint32_t bytes;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(bytes));
        const int slots = (int)(bytes / (sizeof(float4) * blockDim.x));
        const int per = (int)((((N + 3) >> 2) + blockDim.x - 1) / blockDim.x);
        kp.nx = min(slots, per);
        kp.np = min(slots - kp.nx, per);
        kp.x = reinterpret_cast<ulonglong2 *>(us);
        kp.p = kp.x + (int64_t)kp.nx * blockDim.x;
    }
    int start = st->start;
    // sum of the current configuration, carried from trajectory to trajectory
    CSum Sstart = chain_sum<V4>(sel3(A, start) + (int64_t)chain * N, N, red);
    for (int k = 0; k < A.n_traj; ++k) {
        const uint32_t traj = A.traj0 + (uint32_t)k;
        Acc acc = acc_zero();
        CSum cs = Sstart;
        const int prop = buf_loc(start, S.n_pass - 1);
        // the integrator's force passes; the first draws the momenta (Sec. 3
        // refresh), the last evaluates the proposal's action
        for (int j = 0; j < S.n_pass; ++j) {
            PassCfg pc;
            pc.src = j == 0 ? start : prop;
            pc.dst = prop;
            pc.kick = (float)(S.kick[j] * prm.eps);
            pc.drift = (float)(S.drift[j] * prm.eps);
            pc.traj = traj;
            const bool first = j == 0, last = j == S.n_pass - 1;
            if (first && last) inf_pass<V4, true, true>(A, pc, kc, chain, kp, cs, red, tab_s, acc);
            else if (first) inf_pass<V4, true, false>(A, pc, kc, chain, kp, cs, red, tab_s, acc);
            else if (last) inf_pass<V4, false, true>(A, pc, kc, chain, kp, cs, red, tab_s, acc);
            else inf_pass<V4, false, false>(A, pc, kc, chain, kp, cs, red, tab_s, acc);
        }
        double v[7];
        acc_totals(acc, v, red);
        const int cur = metropolis(A, st, prm, chain, traj, start, prop, v, invN, bcast);
        if (cur != start) Sstart = cs;   // accepted: the proposal's sum
        start = cur;
        // ---- optional global sign flip psi -> -psi (Sec. 3, ergodicity) ----
        if (A.flip_every > 0 && ((traj + 1) % (uint32_t)A.flip_every) == 0) {
            Acc fa = acc_zero();
            inf_action<V4>(A, kc, chain, start, -1.0f, traj, kc.rk, red, tab_s, fa);
            double w[5];
            action_totals(fa, w, red);
            if (flip_decision(A, st, prm, chain, traj, w, invN, bcast)) {
                // -psi goes to the buffer that is neither current nor the
                // proposal, so the MD end point stays readable; every thread
                // writes its own quads, as in the resident variant
                const int f = (start != prop) ? 3 - start - prop : (start + 1) % 3;
                const float *gs = sel3(A, start) + (int64_t)chain * N;
                float *gf = sel3(A, f) + (int64_t)chain * N;
                for (int64_t q = threadIdx.x; q < ((N + 3) >> 2); q += blockDim.x) {
                    stq<V4>(gf, 4 * q, N, quad_neg(ldq<V4>(gs, 4 * q, N)));
                }
                start = f;
                Sstart = csum_neg(Sstart);   // negation is exact in every partial sum
                if (threadIdx.x == 0) st->start = f;
            }
            __syncthreads();
        }
        measure(A, st, traj);
    }
}

}  // namespace

// Threads per CTA: one per site quad up to INF_MAX_THREADS, a multiple of 32.
// Fixed by N alone, so the order of every block sum (and with it every
// result) depends on nothing but the model.
int infinite_threads(int64_t N) {
    const int64_t nq = (N + 3) / 4;
    int64_t t = (nq + 31) / 32 * 32;
    if (t > INF_MAX_THREADS) t = INF_MAX_THREADS;
    if (t < 32) t = 32;
    return (int)t;
}

// Quads per thread of the resident variant, or 0 (streaming) when a chain
// needs more than 8 per thread.
static int infinite_qpt(int64_t N) {
    const int64_t nq = (N + 3) / 4;
    const int64_t t = infinite_threads(N);
    for (int q : {1, 2, 4, 8})
        if (nq <= (int64_t)q * t) return q;
    return 0;
}

template <bool V4, bool FULL = false>
static void *infinite_func(int qpt) {
    switch (qpt) {
        case 1: return reinterpret_cast<void *>(infinite_kernel<V4, 1, FULL>);
        case 2: return reinterpret_cast<void *>(infinite_kernel<V4, 2, FULL>);
        case 4: return reinterpret_cast<void *>(infinite_kernel<V4, 4, FULL>);
        case 8: return reinterpret_cast<void *>(infinite_kernel<V4, 8, FULL>);
        default: return reinterpret_cast<void *>(infinite_kernel<V4, 0>);
    }
}

// Slots (a quad of every thread, 4 KB each) of the streaming variant's kept quads: what
// fits beside the 19 KB of static arrays with two CTAs on an SM, or with one
// where the launch has no second one for it.
constexpr int INF_SLOTS_TWO = 23, INF_SLOTS_ONE = 51;
constexpr size_t INF_SLOT_BYTES = INF_MAX_THREADS * sizeof(float4);
constexpr size_t INF_STATIC_BYTES = LOG1PEXP_NODES * sizeof(float4) + 1024;
static_assert(INF_SLOTS_TWO * INF_SLOT_BYTES + INF_STATIC_BYTES <= 113 * 1024, "two CTAs per SM");
static_assert(INF_SLOTS_ONE * INF_SLOT_BYTES + INF_STATIC_BYTES <= 227 * 1024, "one CTA per SM");

static size_t infinite_kept_bytes(int64_t N, int chains) {
    const int sms = sm_count();
    const int64_t per = ((N + 3) / 4 + INF_MAX_THREADS - 1) / INF_MAX_THREADS;
    const int64_t slots = chains <= sms ? INF_SLOTS_ONE : INF_SLOTS_TWO;
    return (size_t)(slots < 2 * per ? slots : 2 * per) * INF_SLOT_BYTES;
}

cudaError_t infinite_node(const FusedArgs &a, cudaKernelNodeParams *np, void **args) {
    const int qpt = infinite_qpt(a.g.N);
    const int64_t nq = (a.g.N + 3) / 4;
    const bool full = a.g.N % 4 == 0 && qpt > 0 && qpt <= 4 && nq == (int64_t)qpt * infinite_threads(a.g.N);
    np->func = full ? infinite_func<true, true>(qpt)
                    : (a.g.N % 4 == 0) ? infinite_func<true>(qpt) : infinite_func<false>(qpt);
    // room for the largest arrays above the static ones, once per device
    static DeviceOnce once;
    int dev = 0;
    const cudaError_t ed = cudaGetDevice(&dev);
    if (ed != cudaSuccess) return ed;
    const cudaError_t es = once.run(dev, [] {
        for (int q : {0, 1, 2, 4, 8})
            for (void *f : {infinite_func<true>(q), infinite_func<false>(q), infinite_func<true, true>(q)}) {
                const cudaError_t e = cudaFuncSetAttribute(
                    f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                    q ? 2 * 8 * INF_MAX_THREADS * 16 : (int)(INF_SLOTS_ONE * INF_SLOT_BYTES));
                if (e != cudaSuccess) return e;
            }
        return cudaSuccess;
    });
    if (es != cudaSuccess) return es;
    np->gridDim = dim3((unsigned)(a.n_chains - a.chain0), 1, 1);
    np->blockDim = dim3((unsigned)infinite_threads(a.g.N), 1, 1);
    // u and aux of the resident variant: at most 2 x 8 quads x 256 threads x 16 B = 64 KB;
    // the streaming variant's kept quads
    np->sharedMemBytes = qpt ? (unsigned)(2 * qpt * infinite_threads(a.g.N) * sizeof(float4))
                             : (unsigned)infinite_kept_bytes(a.g.N, a.n_chains - a.chain0);
    np->kernelParams = args;
    np->extra = nullptr;
    return cudaSuccess;
}

cudaError_t launch_infinite(const FusedArgs &a, const Schedule &sched, cudaStream_t s) {
    cudaKernelNodeParams np;
    void *args[2] = {const_cast<FusedArgs *>(&a), const_cast<Schedule *>(&sched)};
    cudaError_t e = infinite_node(a, &np, args);
    if (e != cudaSuccess) return e;
    if (np.gridDim.x == 0) return cudaSuccess;
    return cudaLaunchKernel(np.func, np.gridDim, np.blockDim, np.kernelParams, np.sharedMemBytes, s);
}

}  // namespace ihmc
