// k_rates3.cuh - parts shared by the three-phonon rate and adjoint kernels: the cluster sums G of a
// mode, the window of a round of partner points with the queue of kept processes, and V3 of one process.
#pragma once
#include "fc4_window.cuh"

namespace fc4 {

constexpr int kR3Threads = 128;

// partner branches j' tested per compaction (JB; bounds the queue: kR3Threads * (JB * nb + 1) entries)
constexpr int jb3(int nb) { return nb <= 6 ? nb : nb <= 12 ? 3 : 1; }

// A queued process is one word: q' - qlo in its upper 16 bits, j' and j'' in 8 each.  A queue therefore holds
// partner points [qlo, qlo + kQueueSpan3) only.
constexpr int kQueueSpan3 = 1 << 16;

// One mode λ = (q0, j0) and channel sign s: q'' = q + s q'.
struct Three {
    int ch, s, m0, q0, j0;
    int4 c0;
    double w0;
    float w0f;
    __device__ __forceinline__ Three(const Tables &t, int ch_, int m, int nb)
        : ch(ch_), s(ch_ == 0 ? 1 : -1), m0(m), q0(m / nb), j0(m - (m / nb) * nb), c0(t.qc[m / nb]),
          w0(t.om[m]), w0f(t.om32[m]) {}
};

// G_r[βγ] = Σ_{clusters in r} exp(-i q.R2) / sqrt(m) Σ_α Φ[αβγ] e_λ(aα) into sG [n_keys3][9], by key or (PERM) in the
// FP64 key order; se0: e_λ in shared memory.
template <bool PERM>
__device__ __forceinline__ void three_G(const Tables &t, const Three &p, const double2 *se0, double2 *sG) {
    for (int k = threadIdx.x; k < t.n_keys3 * 9; k += kR3Threads) {
        const int r = k / 9, bg = k - 9 * r;
        double2 g = czero<double2>();
        for (int i = t.k3_start[r]; i < t.k3_start[r + 1]; ++i) {
            const int c = t.k3_idx[i], a0 = t.c3_at[c].x;
            const double *phi = t.phi3 + 27 * c + bg;
            double2 v = czero<double2>();
#pragma unroll
            for (int al = 0; al < 3; ++al) v = crfma(phi[9 * al], se0[3 * a0 + al], v);
            const double2 ph = cconj(t.rt[phase_index(p.c0, t.c3_r2[c], t.L)]);
            g = cfma(cmake(ph.x * t.c3_ism[c], ph.y * t.c3_ism[c]), v, g);
        }
        sG[PERM ? 9 * t.pos3[r] + bg : k] = g;
    }
}

// Window of the partner points qb + thread (below qhi <= qlo + kQueueSpan3) and branches jb .. jb + JB - 1 against every
// j'': the kept processes (q' - qlo, j', j'') are appended in order to sList at queued.  Returns the new
// length.  Ends with a block barrier.
template <int NB, bool ADA, int JB>
__device__ __forceinline__ int three_append(const Tables &t, const RateArgs &a, const Three &p, int qlo, int qb,
                                            int qhi, int jb, int queued, unsigned *sList, int *s_scan) {
    const int q1 = qb + threadIdx.x;
    int q2 = 0;
    unsigned v1 = 0, v2 = 0;
    if (q1 < qhi) {
        const int4 c1 = t.qc[q1];
        q2 = q_index(p.c0.x + p.s * c1.x, p.c0.y + p.s * c1.y, p.c0.z + p.s * c1.z, t.mesh[0], t.mesh[1], t.mesh[2]);
        v1 = t.vmask[q1];
        v2 = t.vmask[q2];
    }
    unsigned kept[JB];
    int n = 0;
#pragma unroll
    for (int jj = 0; jj < JB; ++jj) {
        const int j1 = jb + jj;
        kept[jj] = 0;
        if (!((v1 >> j1) & 1u)) continue;
        const float base32 = p.w0f + (float)p.s * t.om32[q1 * NB + j1];
        const int m1 = q1 * NB + j1;
        for (int j2 = 0; j2 < NB; ++j2) {
            if (!((v2 >> j2) & 1u)) continue;
            const int m2 = q2 * NB + j2;
            const float ad = fabsf(base32 - t.om32[m2]);
            bool keep;
            if constexpr (ADA) {
                const int w = window_adaptive32(a, ad, two_sigma32(t, a, m1, m2));
                keep = w == 2 || (w == 1 && window_exact_adaptive(t, a, p.ch, p.m0, m1, m2, -1, m1, m2));
            } else {
                if (ad <= a.lo32) keep = true;
                else if (ad > a.hi32) keep = false;
                else keep = fabs(delta_exact(p.ch, p.w0, t.om[m1], t.om[m2], 0.0)) <= a.two_sigma;
            }
            kept[jj] |= (unsigned)keep << j2;
        }
        n += __popc(kept[jj]);
    }
    int total;
    int off = queued + block_exclusive_scan(n, s_scan, &total);
#pragma unroll
    for (int jj = 0; jj < JB; ++jj) {
        unsigned m = kept[jj];
        while (m) {
            const int j2 = __ffs(m) - 1;
            m &= m - 1;
            sList[off++] = ((unsigned)(q1 - qlo) << 16) | ((unsigned)(jb + jj) << 8) | (unsigned)j2;
        }
    }
    __syncthreads();
    return queued + total;
}

// A queued process: its partner modes, V3 and its weight (symmetry, occupations, Gaussian, 1/Πω).
struct ThreeProcess {
    int q1, q2, j1, j2, m1, m2;
    double2 V;
    double w;
};

template <int NA, bool ADA>
__device__ __forceinline__ ThreeProcess three_evaluate(const Tables &t, const RateArgs &a, const Three &p, int qlo,
                                                       unsigned e, const double2 *sG) {
    constexpr int NB = 3 * NA;
    ThreeProcess z;
    z.q1 = qlo + (int)(e >> 16);
    z.j1 = (int)((e >> 8) & 0xff);
    z.j2 = (int)(e & 0xff);
    const int4 cc1 = t.qc[z.q1];
    z.q2 = q_index(p.c0.x + p.s * cc1.x, p.c0.y + p.s * cc1.y, p.c0.z + p.s * cc1.z, t.mesh[0], t.mesh[1], t.mesh[2]);
    z.m1 = z.q1 * NB + z.j1;
    z.m2 = z.q2 * NB + z.j2;
    const double2 *P = t.P3 + (size_t)z.q1 * t.n_keys3;
    const double2 *e1p = t.ev + (size_t)z.q1 * NB * NB + z.j1, *e2p = t.ev + (size_t)z.q2 * NB * NB + z.j2;
    z.V = czero<double2>();
#pragma unroll 1
    for (int b = 0; b < NA; ++b)
#pragma unroll 1
        for (int c = 0; c < NA; ++c) {
            const int r0 = t.grp3_start[b * NA + c], r1 = t.grp3_start[b * NA + c + 1];
            if (r0 == r1) continue;
            double2 T[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) T[k] = czero<double2>();
#pragma unroll 1
            for (int r = r0; r < r1; ++r) {
                const double2 ph = cconj_if(P[r], p.s < 0);
                const double2 *G = sG + 9 * r;
#pragma unroll
                for (int k = 0; k < 9; ++k) T[k] = cfma(ph, G[k], T[k]);
            }
            double2 e2[3];
#pragma unroll
            for (int g = 0; g < 3; ++g) e2[g] = cconj(e2p[(3 * c + g) * NB]);
#pragma unroll
            for (int be = 0; be < 3; ++be) {
                double2 u = cmul(T[3 * be], e2[0]);
                u = cfma(T[3 * be + 1], e2[1], u);
                u = cfma(T[3 * be + 2], e2[2], u);
                z.V = cfma(cconj_if(e1p[(3 * b + be) * NB], p.s < 0), u, z.V);
            }
        }
    const double d = delta_exact(p.ch, p.w0, t.om[z.m1], t.om[z.m2], 0.0);
    double g;
    if constexpr (ADA) g = gauss_adaptive(t, a, d, z.m1, z.m2);
    else g = exp(-(d * d) * a.inv_sigma2) * a.gnorm;
    z.w = (p.ch == 0 ? 1.0 : 0.5) * occupation_factor<double>(p.ch, t.occ[z.m1], t.occ[z.m2], 0.0) * g *
          t.invw[p.m0] * t.invw[z.m1] * t.invw[z.m2];
    return z;
}

}  // namespace fc4
