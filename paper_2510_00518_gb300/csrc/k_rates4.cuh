// k_rates4.cuh - fused four-phonon kernel: enumeration, energy window, matrix element V4,
// weight and per-(λ, q') reduction, for one channel (++, +-, --).
//
// The paper (Algorithms 3-4) enumerates the kept processes on the CPU, ships index lists to
// the GPU and evaluates V per process.  Here the same work is fused and factored so that the
// dense parts are shared.  One thread block owns a unit (λ = (q, j), q') and loops over the
// partner branch j'.  With q''' = q + s1 q' + s2 q'', the phase of a cluster factorises as
//   exp(i(s1 q'.R1 + s2 q''.R2 - q'''.R3)) = exp(-i q.R3) exp(i s1 q'.(R1 - R3)) exp(i s2 q''.(R2 - R3)),
// so with a "key" r = (leg-2 atom c, leg-3 atom d, R2 - R3) the element is
//   V = Σ_r P_r(q'')^s2 Σ_γδ W_r[γδ] e^s2_λ''(cγ) e*_λ'''(dδ),
//   W_r[γδ] = Σ_{clusters in r} exp(-i q.R3 + i s1 q'.(R1 - R3)) / sqrt(m) Σ_αβ Φ[αβγδ] e_λ(aα) e^s1_λ'(bβ),
// W built once per (λ, q', j') in shared memory.  Partners q'' are enumerated one per thread,
// the window is tested with an FP32 prefilter of proven error bound (ambiguous cases are
// decided by the exact FP64 Δ), kept (q'', j''', j''-mask) items are compacted in order by a
// block scan, and each item computes Y[cγ] = Σ_r P_r Σ_δ W_r[γδ] e*_λ'''(dδ) once for all its
// j'' (V = Σ_cγ e^s2_λ''(cγ) Y[cγ]).
#pragma once
#include <algorithm>

#include "fc4_window.cuh"

namespace fc4 {

template <typename R>
struct Sel {
    static __device__ __forceinline__ const Cplx<R> *ev(const Tables &t);
    static __device__ __forceinline__ const Cplx<R> *rt(const Tables &t);
    static __device__ __forceinline__ const Cplx<R> *P4(const Tables &t);
    static __device__ __forceinline__ const R *phi4(const Tables &t);
    static __device__ __forceinline__ const R *ism4(const Tables &t);
    static __device__ __forceinline__ const R *occ(const Tables &t);
    static __device__ __forceinline__ const R *invw(const Tables &t);
    static __device__ __forceinline__ const R *om(const Tables &t);
    static __device__ __forceinline__ const R *bteF(const RateArgs &a);
};
template <> struct Sel<double> {
    static __device__ __forceinline__ const double2 *ev(const Tables &t) { return t.ev; }
    static __device__ __forceinline__ const double2 *rt(const Tables &t) { return t.rt; }
    static __device__ __forceinline__ const double2 *P4(const Tables &t) { return t.P4; }
    static __device__ __forceinline__ const double *phi4(const Tables &t) { return t.phi4; }
    static __device__ __forceinline__ const double *ism4(const Tables &t) { return t.c4_ism; }
    static __device__ __forceinline__ const double *occ(const Tables &t) { return t.occ; }
    static __device__ __forceinline__ const double *invw(const Tables &t) { return t.invw; }
    static __device__ __forceinline__ const double *om(const Tables &t) { return t.om; }
    static __device__ __forceinline__ const double *bteF(const RateArgs &a) { return a.bte_F; }
};
template <> struct Sel<float> {
    static __device__ __forceinline__ const float2 *ev(const Tables &t) { return t.ev32; }
    static __device__ __forceinline__ const float2 *rt(const Tables &t) { return t.rt32; }
    static __device__ __forceinline__ const float2 *P4(const Tables &t) { return t.P4_32; }
    static __device__ __forceinline__ const float *phi4(const Tables &t) { return t.phi4_32; }
    static __device__ __forceinline__ const float *ism4(const Tables &t) { return t.c4_ism32; }
    static __device__ __forceinline__ const float *occ(const Tables &t) { return t.occ32; }
    static __device__ __forceinline__ const float *invw(const Tables &t) { return t.invw32; }
    static __device__ __forceinline__ const float *om(const Tables &t) { return t.om32; }
    static __device__ __forceinline__ const float *bteF(const RateArgs &a) { return a.bte_F32; }
};

// Exact FP64 decision for the rare candidates inside the prefilter's ambiguity band (kept out of
// line: the unrolled branch loops stay small).
static __device__ __noinline__ bool window_exact4(int ch, double w0, double w1, double w2, double w3,
                                            double two_sigma) {
    return fabs(delta_exact(ch, w0, w1, w2, w3)) <= two_sigma;
}

// symmetry factor of the 4ph channels: 1/2 (++, +-), 1/6 (--)
template <typename R> __device__ __forceinline__ R sym4(int ch) { return ch == 4 ? R(1) / R(6) : R(0.5); }

constexpr int kQChunk = 1024;      // partner q'' handled per compaction round

// Error-free sum: a + b = s + e exactly (Knuth's TwoSum, round-to-nearest FP32).
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
    const float s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}

// Δ = ω + s1 ω' + s2 ω'' - ω''' from hi/lo FP32 splits of each ω (|error| ~ 2^-44 ω_max): the
// Gaussian's argument in the mixed path without FP64 instructions.
__device__ __forceinline__ float delta_comp(float h0, float l0, float h1, float l1, float h2, float l2,
                                            float h3, float l3, int s1, int s2) {
    float e1, e2, e3;
    const float x1 = two_sum(h0, (float)s1 * h1, e1);
    const float x2 = two_sum(x1, (float)s2 * h2, e2);
    const float x3 = two_sum(x2, -h3, e3);
    const float lo = ((l0 + (float)s1 * l1) + ((float)s2 * l2 - l3));
    return x3 + ((e1 + e2) + (e3 + lo));
}

// Triangular domain of a (q', q'') pair (partner-swap symmetry of the summand): -1 the pair is the
// swap of one evaluated elsewhere; 0 no symmetry used (weight 1); 1 weight 2; 2 +- with q'' = q'''
// (keep j'' <= j'''); 3 ++ / -- with q'' = q' (keep j'' >= j').  domains: bits as RateArgs::tri.
__device__ __forceinline__ int tri_code(int domains, int ch, int q1, int q2, int q3) {
    if (ch == 3) {
        if (!(domains & 1)) return 0;
        return q2 > q3 ? -1 : (q2 < q3 ? 1 : 2);
    }
    if (!(domains & 2)) return 0;
    return q2 < q1 ? -1 : (q2 > q1 ? 1 : 3);
}

// tri_code of a (q', q'') pair of mode m0 under the sampling estimate: a representative stands for
// its own pair and, off the diagonal (code 1), for its swapped pair ((λ, q', q''') for +-,
// (λ, q'', q') for ++ and --); it keeps weight 2 when both are in the sample, becomes weight 1
// (code 0) when one is, and is skipped (-1) when neither is.
__device__ __forceinline__ int tri_code_sampled(const RateArgs &a, int domains, int ch, int m0, int q1, int q2, int q3,
                                                int N) {
    const int tri = tri_code(domains, ch, q1, q2, q3);
    if (a.sample_all || tri < 0) return tri;
    const int sa = pair_sampled(a, m0, q1, q2, N) ? 1 : 0;
    if (tri != 1) return sa ? tri : -1;
    const int sb = (ch == 3 ? pair_sampled(a, m0, q1, q3, N) : pair_sampled(a, m0, q2, q1, N)) ? 1 : 0;
    return sa + sb == 2 ? 1 : sa + sb == 1 ? 0 : -1;
}

__device__ __forceinline__ int tri_code_sampled(const RateArgs &a, int ch, int m0, int q1, int q2, int q3, int N) {
    return tri_code_sampled(a, a.tri, ch, m0, q1, q2, q3, N);
}

// weight of an evaluated process: 2 for a swapped pair, 1 on the diagonal or without symmetry
__device__ __forceinline__ int tri_weight(int tri, int j1, int j2, int j3) {
    return tri == 0 ? 1 : tri == 1 ? 2 : tri == 2 ? (j2 < j3 ? 2 : 1) : (j2 > j1 ? 2 : 1);
}

// Window masks of one q'': bit j'' of mask[j'''] is set iff the process is kept (restricted to the
// triangular domain).  FP32 prefilter with the proven bound; candidates inside the band are
// decided by the exact FP64 Δ.
template <int NB, bool ADA>
__device__ __forceinline__ int window_masks(const Tables &t, const RateArgs &a, int domains, int ch, int s2,
                                            float base32, int m0, int m1, double w0, double w1, int q2,
                                            int q3, unsigned (&mask)[NB]) {
    const unsigned v2 = t.vmask[q2], v3 = t.vmask[q3];
    const int q1 = m1 / NB, j1 = m1 - q1 * NB;
    const int tri = tri_code_sampled(a, domains, ch, m0, q1, q2, q3, t.N);
    // no pair of the point can reach the window: FP32 sums are monotonic, and no width exceeds the one of
    // |P''| + |P'''|
    const float4 r2 = t.wrange[q2], r3 = t.wrange[q3];
    const float thr = ADA ? fmaf(a.ad_rhi, a.ad_c32 * (r2.z + r3.z), a.ad_e0) : a.hi32;
    const bool out = (base32 + (s2 > 0 ? r2.x : -r2.y)) - r3.y > thr || (base32 + (s2 > 0 ? r2.y : -r2.x)) - r3.x < -thr;
    if (tri < 0 || out) {
#pragma unroll
        for (int j3 = 0; j3 < NB; ++j3) mask[j3] = 0u;
        return 0;
    }
    // branch pairs of the domain: j'' <= j''' (tri 2) or j'' >= j' (tri 3)
    auto dom = [&](int j3) -> unsigned {
        return tri == 2 ? (2u << j3) - 1u : tri == 3 ? ~((1u << j1) - 1u) : ~0u;
    };
    if constexpr (ADA) {
        int n = 0;
        for (int j3 = 0; j3 < NB; ++j3) {
            mask[j3] = ((v3 >> j3) & 1u) ? window_adaptive4_row<NB>(t, a, ch, s2, base32, m0, m1, q2, q3, j3, v2) & dom(j3)
                                         : 0u;
            n += (mask[j3] != 0);
        }
        return n;
    }
    float t2[NB], w3f[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        t2[j] = base32 + (float)s2 * t.omT32[(size_t)j * t.N + q2];
        w3f[j] = t.omT32[(size_t)j * t.N + q3];
    }
    int n = 0;
#pragma unroll
    for (int j3 = 0; j3 < NB; ++j3) {
        unsigned m = 0;
        if ((v3 >> j3) & 1u) {
#pragma unroll
            for (int j2 = 0; j2 < NB; ++j2) {
                if (!((v2 >> j2) & 1u)) continue;
                const float ad = fabsf(t2[j2] - w3f[j3]);
                bool keep;
                if (ad <= a.lo32) keep = true;
                else if (ad > a.hi32) keep = false;
                else keep = window_exact4(ch, w0, w1, t.om[q2 * NB + j2], t.om[q3 * NB + j3], a.two_sigma);
                m |= (unsigned)keep << j2;
            }
        }
        mask[j3] = m & dom(j3);
        n += (mask[j3] != 0);
    }
    return n;
}

// One row of the window of (λ, λ'; q''): bit j'' set iff the process with λ''' = (q3, j3) is kept,
// restricted to the triangular domain.  A row none of whose |Δ32| can reach the window (FP32 sums are
// monotonic in ω''; lo2, hi2: range of s2 ω'' over the participating branches; thr bounds the window of
// every pair) is decided without looking at its pairs.
template <int NB, bool ADA>
__device__ __forceinline__ unsigned window_row(const Tables &t, const RateArgs &a, int ch, int s2, float base32,
                                               int m0, int m1, int j1, double w0, int q2, int q3, unsigned v2,
                                               int j3, int tri, float lo2, float hi2, float thr) {
    const float w3 = t.omT32[(size_t)j3 * t.N + q3];
    if ((base32 + lo2) - w3 > thr || (base32 + hi2) - w3 < -thr) return 0u;
    const unsigned dom = tri == 2 ? (2u << j3) - 1u : tri == 3 ? ~((1u << j1) - 1u) : ~0u;
    if constexpr (ADA) {
        return window_adaptive4_row<NB>(t, a, ch, s2, base32, m0, m1, q2, q3, j3, v2) & dom;
    } else {
        unsigned near = 0;
#pragma unroll
        for (int j2 = 0; j2 < NB; ++j2)
            near |= (unsigned)(fabsf((base32 + (float)s2 * t.omT32[(size_t)j2 * t.N + q2]) - w3) <= a.hi32) << j2;
        near &= v2 & dom;
        unsigned m = 0;
        while (near) {
            const int j2 = __ffs(near) - 1;
            near &= near - 1;
            const float ad = fabsf((base32 + (float)s2 * t.omT32[(size_t)j2 * t.N + q2]) - w3);
            if (ad <= a.lo32 || window_exact4(ch, w0, t.om[m1], t.om[q2 * NB + j2], t.om[q3 * NB + j3], a.two_sigma))
                m |= 1u << j2;
        }
        return m;
    }
}

// Kahan-compensated FP32 accumulator (mixed path) / plain FP64 accumulator (FP64 path).
template <typename R> struct Acc {
    double s = 0.0;
    __device__ __forceinline__ void add(R x) { s += (double)x; }
    __device__ __forceinline__ double value() const { return s; }
};
template <> struct Acc<float> {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) {
        const float y = x - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// Shared memory of the general kernel (dynamic).  W of one j' is built in pieces of as many clusters as
// the evaluation's buffers hold; both phases share that space.
constexpr int kSubBatch = 64;      // entries expanded into items at a time
template <typename R, int NA>
struct GeneralSmem {
    using C = Cplx<R>;
    static constexpr int NB = 3 * NA;
    static constexpr bool XROUTE = NA <= 2;
    C *W, *Ph, *E, *e0, *Con;
    unsigned long long *Q;         // X route: entries (q'', masks) [kQChunk]
    unsigned short *ent;           // else: entries (q'') [kQChunk]
    unsigned *found;               // bit per q'' of the chunk
    unsigned *mask;                // [NB][kSubBatch] kept j'' per (j''', entry of the sub-batch)
    unsigned long long *item;      // [kSubBatch * NB]
    R *proc;                       // [128 * NB][2] weight and |V|^2 of a pass' processes
    int n_con;                     // clusters per piece
    __host__ __device__ static size_t buffer_bytes() {
        const size_t ev = XROUTE ? sizeof(unsigned long long) * kQChunk
                                 : sizeof(unsigned) * NB * kSubBatch + sizeof(unsigned long long) * kSubBatch * NB +
                                       2 * sizeof(R) * 128 * NB;
        return ev > 16384 ? ev : 16384;
    }
    __host__ __device__ static size_t bytes(const Tables &t) {
        size_t b = sizeof(C) * ((size_t)t.n_keys * 9 + t.nc4 + NA * NA * 9 + NB + (NB & 1)) + buffer_bytes() +
                   (XROUTE ? 0 : sizeof(unsigned short) * kQChunk + kQChunk / 8);
        return (b + 15) & ~size_t(15);
    }
    __device__ __forceinline__ GeneralSmem(unsigned char *smem, const Tables &t) {
        e0 = reinterpret_cast<C *>(smem);                           // [NB]       e_λ
        E = e0 + NB + (NB & 1);                                     // [NA*NA*9]  e_λ(aα) e^s1_λ'(bβ)
        W = E + NA * NA * 9;                                        // [n_keys * 9]
        Ph = W + t.n_keys * 9;                                      // [nc4]      phase of a cluster at (q, q')
        unsigned char *buf = reinterpret_cast<unsigned char *>(
            (reinterpret_cast<size_t>(Ph + t.nc4) + 15) & ~size_t(15));
        Con = reinterpret_cast<C *>(buf);                           // [n_con * 9] per-cluster terms
        n_con = (int)(buffer_bytes() / (9 * sizeof(C)));
        Q = reinterpret_cast<unsigned long long *>(buf);
        item = reinterpret_cast<unsigned long long *>(buf);
        proc = reinterpret_cast<R *>(item + kSubBatch * NB);
        mask = reinterpret_cast<unsigned *>(proc + 2 * 128 * NB);
        ent = reinterpret_cast<unsigned short *>(buf + buffer_bytes());
        found = reinterpret_cast<unsigned *>(ent + kQChunk);
    }
};

// One (λ, q') unit of the general kernel, run by the whole block (the body of rates4_kernel and of
// the batched persistent kernel, which takes its units from a work list over many contexts).
//
// Up to two atoms, X[c,d][γδ] = Σ_r P_r W_r[γδ] is formed once per entry (q'') by the entry's thread, then
// 36 complex multiply-adds per (q'', j''') item.  Larger cells list their entries, expand them into
// items a sub-batch at a time and take one item per thread: an item's Y (12 n_keys complex multiply-
// adds) is the bulk of the work, and entries carry 1 to nb of them.  The weights of a pass go
// through shared memory to the entry's owner thread, which adds them in order, so Γ's bits are those
// of a thread that walks its entries alone.
// Bound: latency of the item work at 3-4 blocks per SM.  One thread per entry walked its items alone (20
// entries on 128 threads at 4^3) and formed the window three times: one q point of 4^3 with eight
// atoms 314 -> 26 ms (three channels), three q points of 5x5x4 with four atoms and adaptive σ 68 -> 24 ms;
// with the channels in one launch and the window rows shared out, 23 and 16 ms.
template <typename R, int NA, bool ADA>
__device__ __forceinline__ void rates4_unit(const Tables &t, const RateArgs &a, int ch, int unit) {
    using C = Cplx<R>;
    using Smem = GeneralSmem<R, NA>;
    constexpr int NB = 3 * NA;
    constexpr bool XROUTE = Smem::XROUTE;
    const int s1 = (ch == 4) ? -1 : 1;
    const int s2 = (ch == 2) ? 1 : -1;
    const int N = t.N;

    extern __shared__ __align__(16) unsigned char smem[];
    const Smem sm(smem, t);
    __shared__ int s_scan[32];
    __shared__ int s_off[XROUTE ? 1 : 129];                     // process offset of each item of a pass
    __shared__ double s_red[2 * 32];
    __shared__ long long s_redn[5 * 32];

    const int ms = unit / N, q1 = unit - ms * N;
    const int m0 = a.modes[ms];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    const C *ev = Sel<R>::ev(t);
    const C *rt = Sel<R>::rt(t);
    const C *P4 = Sel<R>::P4(t);
    const R *phi4 = Sel<R>::phi4(t);
    const R *ism4 = Sel<R>::ism4(t);
    const R *occ = Sel<R>::occ(t);
    const R *invw = Sel<R>::invw(t);

    Acc<R> acc_g, acc_wp;
    long long acc_n = 0, acc_items = 0, acc_ent = 0, acc_ev = 0, acc_cev = 0;

    const bool active = !(q0 == 0 && j0 < 3);
    if (active) {
        const int4 c0 = t.qc[q0], c1 = t.qc[q1];
        const int b0 = c0.x + s1 * c1.x, b1 = c0.y + s1 * c1.y, b2 = c0.z + s1 * c1.z;
        const double w0 = t.om[m0];
        const float w0f = t.om32[m0];
        const unsigned vm1 = t.vmask[q1];
        __syncthreads();                           // batched form: the previous unit is done with Ph
        for (int k = threadIdx.x; k < NB; k += blockDim.x) sm.e0[k] = ev[(q0 * NB + k) * NB + j0];
        for (int c = threadIdx.x; c < t.nc4; c += blockDim.x)
            sm.Ph[c] = rt[mod_pos(s1 * phase_index(c1, t.c4_r13[c], t.L) - phase_index(c0, t.c4_r3[c], t.L), t.L)];

        // weight of one process, times the number of processes it stands for
        auto weight = [&](int m1, double w1, int m2, int m3, int wt) -> R {
            R w;
            if constexpr (sizeof(R) == 8) {
                const double d = delta_exact(ch, w0, w1, t.om[m2], t.om[m3]);
                double g;
                if constexpr (ADA) g = gauss_adaptive(t, a, d, m2, m3);
                else g = exp(-(d * d) * a.inv_sigma2) * a.gnorm;
                w = sym4<double>(ch) * occupation_factor<double>(ch, occ[m1], occ[m2], occ[m3]) *
                    g * invw[m0] * invw[m1] * invw[m2] * invw[m3];
            } else {
                const float4 k0 = t.mode4[m0], k1 = t.mode4[m1], k2 = t.mode4[m2], k3 = t.mode4[m3];
                const float df = delta_comp(k0.x, k0.y, k1.x, k1.y, k2.x, k2.y, k3.x, k3.y, s1, s2);
                float g;
                if constexpr (ADA) g = gauss_adaptive32(t, a, df, m2, m3);
                else g = __expf(-(df * df) * a.inv_sigma2_32) * a.gnorm32;
                w = sym4<float>(ch) * occupation_factor<float>(ch, k1.z, k2.z, k3.z) * g *
                    (k0.w * k1.w) * (k2.w * k3.w);
            }
            w *= (R)wt;
            return w;
        };

        for (int j1 = 0; j1 < NB; ++j1) {
            if (!((vm1 >> j1) & 1u)) continue;
            const int m1 = q1 * NB + j1;
            __syncthreads();                       // previous j1 finished with the shared tables
            for (int k = threadIdx.x; k < NA * NA * 9; k += blockDim.x) {
                const int ab = k / 9, ij = k - ab * 9;
                const int at = ab / NA, bt = ab - at * NA;
                const int al = ij / 3, be = ij - al * 3;
                C y = cconj_if(ev[(q1 * NB + 3 * bt + be) * NB + j1], s1 < 0);
                sm.E[k] = cmul(sm.e0[3 * at + al], y);
            }
            // W_r[γδ]: per-cluster terms exp(-i q.R3 + i s1 q'.(R1 - R3)) / sqrt(m) Σ_αβ Φ[αβγδ] E[αβ] of a
            // piece, added to their keys in cluster order (deterministic)
            for (int cb = 0; cb < t.nc4; cb += sm.n_con) {
                const int ce = min(t.nc4, cb + sm.n_con);
                __syncthreads();
                for (int k = threadIdx.x; k < (ce - cb) * 9; k += blockDim.x) {
                    const int c = cb + k / 9, gd = k % 9;
                    const int4 at = t.c4_at[c];
                    const R *ph4 = phi4 + 81 * c + gd;
                    const C *E = sm.E + (at.x * NA + at.y) * 9;
                    C v = czero<C>();
#pragma unroll
                    for (int ab = 0; ab < 9; ++ab) v = crfma(ph4[9 * ab], E[ab], v);
                    const C p = cmul(sm.Ph[c], v);
                    sm.Con[k] = cmake(p.x * ism4[c], p.y * ism4[c]);
                }
                __syncthreads();
                for (int k = threadIdx.x; k < t.n_keys * 9; k += blockDim.x) {
                    const int r = k / 9, gd = k - r * 9;
                    C acc = cb ? sm.W[k] : czero<C>();
                    for (int c = max(cb, t.key_start[r]); c < min(ce, t.key_start[r + 1]); ++c)
                        acc = cadd(acc, sm.Con[(c - cb) * 9 + gd]);
                    sm.W[k] = acc;
                }
            }
            __syncthreads();

            const float base32 = w0f + (float)s1 * t.om32[m1];
            const double w1 = t.om[m1];
            // ++ and -- on their triangle (q'' >= q') start at q'' = q'
            for (int qb = (ch != 3 && (a.tri & 2)) ? q1 : 0; qb < N; qb += kQChunk) {
                const int qe = min(N, qb + kQChunk);
                int total;
                if constexpr (XROUTE) {
                    // window masks of this thread's q''; those with a kept process go to the entry list (q''
                    // packed with the 36 mask bits)
                    constexpr int kPer = kQChunk / 64;              // blockDim >= 64
                    unsigned long long ent[kPer];
                    int n_act = 0;
                    for (int q2 = qb + threadIdx.x; q2 < qe; q2 += blockDim.x) {
                        const int4 c2 = t.qc[q2];
                        const int q3 = q_index(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z,
                                               t.mesh[0], t.mesh[1], t.mesh[2]);
                        unsigned mask[NB];
                        if (tri_code_sampled(a, ch, m0, q1, q2, q3, N) >= 0) acc_cev += NB * NB;   // visited
                        if (window_masks<NB, ADA>(t, a, a.tri, ch, s2, base32, m0, m1, w0, w1, q2, q3, mask) > 0) {
                            unsigned long long e = (unsigned long long)q2 << 40;
#pragma unroll
                            for (int j3 = 0; j3 < NB; ++j3) e |= (unsigned long long)mask[j3] << (NB * j3);
                            ent[n_act++] = e;
                        }
                    }
                    const int off = block_exclusive_scan(n_act, s_scan, &total);
                    for (int k = 0; k < n_act; ++k) sm.Q[off + k] = ent[k];
                    __syncthreads();

                    for (int it = threadIdx.x; it < total; it += blockDim.x) {
                        ++acc_ent;
                        const unsigned long long e = sm.Q[it];
                        const int iq2 = (int)(e >> 40);
                        const int4 c2 = t.qc[iq2];
                        const int q3 = q_index(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z,
                                               t.mesh[0], t.mesh[1], t.mesh[2]);
                        const int tri = tri_code_sampled(a, ch, m0, q1, iq2, q3, N);
                        const C *P = P4 + (size_t)iq2 * t.n_keys;
                        C X[NA][NA][9];
#pragma unroll
                        for (int c = 0; c < NA; ++c)
#pragma unroll
                            for (int d = 0; d < NA; ++d) {
#pragma unroll
                                for (int k = 0; k < 9; ++k) X[c][d][k] = czero<C>();
                                const int r0 = t.grp_start[c * NA + d], r1 = t.grp_start[c * NA + d + 1];
                                for (int r = r0; r < r1; ++r) {
                                    const C ph = cconj_if(P[r], s2 < 0);
                                    const C *Wr = sm.W + 9 * r;
#pragma unroll
                                    for (int k = 0; k < 9; ++k) X[c][d][k] = cfma(ph, Wr[k], X[c][d][k]);
                                }
                            }
                        unsigned rows = 0;                          // each lane goes through its own items
#pragma unroll
                        for (int j3 = 0; j3 < NB; ++j3)
                            if ((unsigned)(e >> (NB * j3)) & ((1u << NB) - 1u)) rows |= 1u << j3;
                        while (rows) {
                            const int j3 = __ffs(rows) - 1;
                            rows &= rows - 1;
                            unsigned m = (unsigned)(e >> (NB * j3)) & ((1u << NB) - 1u);
                            ++acc_items;
                            C Y[NA][3];
#pragma unroll
                            for (int c = 0; c < NA; ++c)
#pragma unroll
                                for (int g = 0; g < 3; ++g) Y[c][g] = czero<C>();
                            // Y[cγ] = Σ_dδ X[c,d][γδ] e*_λ'''(dδ)
#pragma unroll
                            for (int d = 0; d < NA; ++d) {
                                C e3[3];
#pragma unroll
                                for (int dl = 0; dl < 3; ++dl) e3[dl] = cconj(ev[(q3 * NB + 3 * d + dl) * NB + j3]);
#pragma unroll
                                for (int c = 0; c < NA; ++c)
#pragma unroll
                                    for (int g = 0; g < 3; ++g)
#pragma unroll
                                        for (int dl = 0; dl < 3; ++dl) Y[c][g] = cfma(X[c][d][3 * g + dl], e3[dl], Y[c][g]);
                            }
                            const int m3 = q3 * NB + j3;
                            while (m) {
                                const int j2 = __ffs(m) - 1;
                                m &= m - 1;
                                C V = czero<C>();
#pragma unroll
                                for (int c = 0; c < NA; ++c)
#pragma unroll
                                    for (int g = 0; g < 3; ++g)
                                        V = cfma(cconj_if(ev[(iq2 * NB + 3 * c + g) * NB + j2], s2 < 0), Y[c][g], V);
                                const int wt = tri_weight(tri, j1, j2, j3);
                                const R w = weight(m1, w1, iq2 * NB + j2, m3, wt);
                                acc_wp.add(w);
                                acc_g.add(w * (V.x * V.x + V.y * V.y));
                                acc_n += wt;
                                acc_ev += 1;
                            }
                        }
                    }
                } else {
                    // closure, domain and window range of a q''
                    struct Point { int q3, tri; unsigned v2, v3; float lo2, hi2, thr; };
                    auto point = [&](int q2) -> Point {
                        Point z;
                        const int4 c2 = t.qc[q2];
                        z.q3 = q_index(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z, t.mesh[0], t.mesh[1], t.mesh[2]);
                        z.tri = tri_code_sampled(a, ch, m0, q1, q2, z.q3, N);
                        z.v2 = t.vmask[q2];
                        z.v3 = t.vmask[z.q3];
                        const float4 r2 = t.wrange[q2], r3 = t.wrange[z.q3];
                        z.lo2 = s2 > 0 ? r2.x : -r2.y;
                        z.hi2 = s2 > 0 ? r2.y : -r2.x;
                        z.thr = ADA ? fmaf(a.ad_rhi, a.ad_c32 * (r2.z + r3.z), a.ad_e0) : a.hi32;
                        return z;
                    };
                    auto row = [&](const Point &z, int q2, int j3) -> unsigned {
                        return ((z.v3 >> j3) & 1u) ? window_row<NB, ADA>(t, a, ch, s2, base32, m0, m1, j1, w0, q2, z.q3,
                                                                         z.v2, j3, z.tri, z.lo2, z.hi2, z.thr)
                                                   : 0u;
                    };
                    // which q'' are entries: three rows of one q'' a thread at a time, those of
                    // a found one left out (a stale read of its bit costs the rows, no more)
                    for (int k = threadIdx.x; k < kQChunk / 32; k += blockDim.x) sm.found[k] = 0;
                    __syncthreads();
                    for (int k = threadIdx.x; k < (qe - qb) * NA; k += blockDim.x) {
                        const int jg = 3 * (k / (qe - qb)), o = k % (qe - qb), q2 = qb + o;
                        const Point z = point(q2);
                        if (z.tri < 0) continue;
                        acc_cev += 3 * NB;                          // visited
                        if ((reinterpret_cast<volatile unsigned *>(sm.found)[o >> 5] >> (o & 31)) & 1u) continue;
                        if (row(z, q2, jg) || row(z, q2, jg + 1) || row(z, q2, jg + 2))
                            atomicOr(&sm.found[o >> 5], 1u << (o & 31));
                    }
                    __syncthreads();
                    // the list, in the order of a thread per q'' (its first, second, ... q'')
                    unsigned found = 0;
                    int i = 0;
                    for (int o = threadIdx.x; o < qe - qb; o += blockDim.x, ++i)
                        found |= ((sm.found[o >> 5] >> (o & 31)) & 1u) << i;
                    int off = block_exclusive_scan(__popc(found), s_scan, &total);
                    for (; found; found &= found - 1)
                        sm.ent[off++] = (unsigned short)((__ffs(found) - 1) * blockDim.x + threadIdx.x);
                    __syncthreads();

                    const int sub = blockDim.x % kSubBatch ? 32 : kSubBatch;
                    for (int eb = 0; eb < total; eb += sub) {
                        // expand: the rows of the sub-batch over all threads, then the entry's owner (the thread
                        // it % blockDim of the whole list) lists its items
                        const int n_sub = min(sub, total - eb);
                        for (int k = threadIdx.x; k < n_sub * NB; k += blockDim.x) {
                            const int j3 = k / n_sub, o = k - j3 * n_sub, eq2 = qb + sm.ent[eb + o];
                            sm.mask[j3 * kSubBatch + o] = row(point(eq2), eq2, j3);
                        }
                        __syncthreads();
                        const int mine = (int)threadIdx.x - eb % (int)blockDim.x;     // slot in the sub-batch
                        const bool own = mine >= 0 && mine < n_sub;
                        int n_it = 0, q2 = 0, tri = 0;
                        if (own) {
                            ++acc_ent;
                            q2 = qb + sm.ent[eb + mine];
                            tri = point(q2).tri;
#pragma unroll 1
                            for (int j3 = 0; j3 < NB; ++j3) n_it += sm.mask[j3 * kSubBatch + mine] != 0;
                        }
                        int n_items;
                        const int it0 = block_exclusive_scan(n_it, s_scan, &n_items), it1 = it0 + n_it;
                        if (own) {
                            int o = it0;
#pragma unroll 1
                            for (int j3 = 0; j3 < NB; ++j3) {
                                const unsigned m = sm.mask[j3 * kSubBatch + mine];
                                if (m) sm.item[o++] = ((unsigned long long)(unsigned)q2 << 36) | ((unsigned long long)tri << 32) |
                                                      ((unsigned long long)j3 << 24) | m;
                            }
                        }
                        __syncthreads();
                        for (int pb = 0; pb < n_items; pb += blockDim.x) {
                            const int n_pass = min((int)blockDim.x, n_items - pb);
                            unsigned long long e = 0;
                            if ((int)threadIdx.x < n_pass) e = sm.item[pb + threadIdx.x];
                            unsigned m = (unsigned)e & 0xffffffu;
                            int n_proc;
                            int po = block_exclusive_scan(__popc(m), s_scan, &n_proc);
                            if ((int)threadIdx.x < n_pass) s_off[threadIdx.x] = po;
                            if (threadIdx.x == 0) s_off[n_pass] = n_proc;
                            if (m) {
                                ++acc_items;
                                const int iq2 = (int)(e >> 36), itri = (int)((e >> 32) & 3u), j3 = (int)((e >> 24) & 0xffu);
                                const int4 c2 = t.qc[iq2];
                                const int q3 = q_index(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z,
                                                       t.mesh[0], t.mesh[1], t.mesh[2]);
                                const C *P = P4 + (size_t)iq2 * t.n_keys;
                                // Y[cγ] = Σ_d Σ_{r in (c,d)} P_r^s2 Σ_δ W_r[γδ] e*_λ'''(dδ)
                                C Y[NA][3];
#pragma unroll
                                for (int c = 0; c < NA; ++c) {
#pragma unroll
                                    for (int g = 0; g < 3; ++g) Y[c][g] = czero<C>();
#pragma unroll 1
                                    for (int d = 0; d < NA; ++d) {
                                        const int r0 = t.grp_start[c * NA + d], r1 = t.grp_start[c * NA + d + 1];
                                        if (r0 == r1) continue;
                                        C e3[3];
#pragma unroll
                                        for (int dl = 0; dl < 3; ++dl) e3[dl] = cconj(ev[(q3 * NB + 3 * d + dl) * NB + j3]);
                                        for (int r = r0; r < r1; ++r) {
                                            const C ph = cconj_if(P[r], s2 < 0);
                                            const C *Wr = sm.W + 9 * r;
#pragma unroll
                                            for (int g = 0; g < 3; ++g) {
                                                C u = cmul(Wr[3 * g], e3[0]);
                                                u = cfma(Wr[3 * g + 1], e3[1], u);
                                                u = cfma(Wr[3 * g + 2], e3[2], u);
                                                Y[c][g] = cfma(ph, u, Y[c][g]);
                                            }
                                        }
                                    }
                                }
                                const int m3 = q3 * NB + j3;
                                while (m) {
                                    const int j2 = __ffs(m) - 1;
                                    m &= m - 1;
                                    C V = czero<C>();
#pragma unroll
                                    for (int c = 0; c < NA; ++c)
#pragma unroll
                                        for (int g = 0; g < 3; ++g)
                                            V = cfma(cconj_if(ev[(iq2 * NB + 3 * c + g) * NB + j2], s2 < 0), Y[c][g], V);
                                    const int wt = tri_weight(itri, j1, j2, j3);
                                    const R w = weight(m1, w1, iq2 * NB + j2, m3, wt);
                                    sm.proc[2 * po] = w;
                                    sm.proc[2 * po + 1] = V.x * V.x + V.y * V.y;
                                    ++po;
                                    acc_n += wt;
                                    acc_ev += 1;
                                }
                            }
                            __syncthreads();
                            // the owner adds its entry's processes of this pass, in order
                            const int lo = max(it0, pb) - pb, hi = min(it1, pb + n_pass) - pb;
                            if (lo < hi)
                                for (int k = s_off[lo]; k < s_off[hi]; ++k) {
                                    acc_wp.add(sm.proc[2 * k]);
                                    acc_g.add(sm.proc[2 * k] * sm.proc[2 * k + 1]);
                                }
                            __syncthreads();       // proc, s_off and item reused
                        }
                    }
                }
                __syncthreads();                   // the entry list is reused by the next chunk
            }
        }
    }
    double sums[2] = {acc_g.value(), acc_wp.value()};
    long long cnts[5] = {acc_n, acc_items, acc_ent, acc_ev, acc_cev};
    block_sum_multi<2, 5>(sums, cnts, s_red, s_redn);
    if (threadIdx.x == 0) {
        const size_t o = ((size_t)ch * a.n_modes + ms) * N + q1;
        a.part_g[o] = sums[0];
        a.part_wp[o] = sums[1];
        a.part_n[o] = cnts[0];
        a.part_items[o] = cnts[1];
        a.part_ent[o] = cnts[2];
        if (a.part_ev) a.part_ev[o] = cnts[3];
        if (a.part_cev) a.part_cev[o] = cnts[4];
    }
}

// Blocks per SM: 4 (128 registers); FP64 cells of up to two atoms hold X (2 blocks, 255 registers).
template <typename R, int NA> constexpr int general_blocks() { return sizeof(R) == 8 && NA <= 2 ? 2 : 4; }

template <typename R, int NA, bool ADA>
__global__ void __launch_bounds__(128, general_blocks<R, NA>())
rates4_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int channels) {
    rates4_unit<R, NA, ADA>(t, a, (channels >> (4 * blockIdx.y)) & 15, blockIdx.x);
}

template <typename R, int NA, bool ADA>
cudaError_t launch4(const Tables &t, const RateArgs &a, int channels, int threads, cudaStream_t s) {
    const size_t smem = GeneralSmem<R, NA>::bytes(t);
    cudaError_t e = cudaFuncSetAttribute(rates4_kernel<R, NA, ADA>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long units = (long long)a.n_modes * t.N;
    if (units > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    if (units == 0) return cudaSuccess;
    const int n_ch = channels >> 8 ? 3 : channels >> 4 ? 2 : 1;
    rates4_kernel<R, NA, ADA><<<dim3((unsigned)units, n_ch), threads, smem, s>>>(t, a, channels);
    e = cudaGetLastError();
    if (e == cudaSuccess && a.n_kernels) ++*a.n_kernels;
    return e;
}

// Dynamic shared memory of the general kernel for one context's tables.
template <typename R, int NA>
size_t general_smem_bytes(const Tables &t) { return GeneralSmem<R, NA>::bytes(t); }

template <typename R, int NA, int HI>
size_t general_smem_atoms(int na, const Tables &t) {
    if (na == NA) return general_smem_bytes<R, NA>(t);
    if constexpr (NA < HI) return general_smem_atoms<R, NA + 1, HI>(na, t);
    else return 0;
}

// Dispatch over the atom count NA..HI (instantiations split across translation units so that they
// compile in parallel; ADA selects the adaptive-σ window and Gaussian at compile time so that the
// fixed-σ kernels carry none of its registers).
// channels: up to three channels, four bits each from the first down, run by one launch (their blocks
// fill each other's last wave).
template <typename R, bool ADA, int NA, int HI>
cudaError_t launch4_atoms(int na, const Tables &t, const RateArgs &a, int channels, int threads, cudaStream_t s) {
    if (na == NA) return launch4<R, NA, ADA>(t, a, channels, threads, s);
    if constexpr (NA < HI) return launch4_atoms<R, ADA, NA + 1, HI>(na, t, a, channels, threads, s);
    else return cudaErrorInvalidValue;
}

// general-kernel launchers, one per translation unit: precision x adaptive x atoms 1-4 / 5-8
#define FC4_GENERAL_LAUNCHER(name) \
    cudaError_t name(int na, const Tables &t, const RateArgs &a, int channels, int threads, cudaStream_t s);
FC4_GENERAL_LAUNCHER(launch4_d_1_4)
FC4_GENERAL_LAUNCHER(launch4_d_5_8)
FC4_GENERAL_LAUNCHER(launch4_f_1_4)
FC4_GENERAL_LAUNCHER(launch4_f_5_8)
FC4_GENERAL_LAUNCHER(launch4_ad_d_1_4)
FC4_GENERAL_LAUNCHER(launch4_ad_d_5_8)
FC4_GENERAL_LAUNCHER(launch4_ad_f_1_4)
FC4_GENERAL_LAUNCHER(launch4_ad_f_5_8)
#undef FC4_GENERAL_LAUNCHER

// tiled-path launchers (<= 2 atoms)
cudaError_t launch4_tile_f(int na, const Tables &t, const RateArgs &a, int ch, cudaStream_t s);
cudaError_t launch4_tile_d(int na, const Tables &t, const RateArgs &a, int ch, cudaStream_t s);
cudaError_t launch4_tile_ad_f(int na, const Tables &t, const RateArgs &a, int ch, cudaStream_t s);
cudaError_t launch4_tile_ad_d(int na, const Tables &t, const RateArgs &a, int ch, cudaStream_t s);
cudaError_t launch4_tile_bte_f(int na, const Tables &t, const RateArgs &a, int ch, cudaStream_t s);
cudaError_t launch4_tile_bte_d(int na, const Tables &t, const RateArgs &a, int ch, cudaStream_t s);

}  // namespace fc4
