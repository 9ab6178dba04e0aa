// k_rates3.cu - three-phonon kernel (channels 3ph+ and 3ph-), FP64 in both precision modes.
//
// With the key r = (leg-1 atom b, leg-2 atom c, R1 - R2) of a cluster the phase factorises, and
//   V3^s = Σ_r P_r(q')^s Σ_βγ G_r[βγ] e^s_λ'(bβ) e*_λ''(cγ),   P_r = exp(i q'.(R1 - R2)),
//   G_r[βγ] = Σ_{clusters in r} exp(-i q.R2) / sqrt(m) Σ_α Φ[αβγ] e_λ(aα)
// (the phase of exp(i(s q'.R1 - q''.R2)) with q'' = q + s q').  One block owns a mode λ and a span
// of kSpan3 partner points q'.  It builds G once in shared memory (two-atom diamond: 98 clusters
// fold into 34 keys), tests the window branch by branch (FP32 prefilter of proven bound, exact FP64
// Δ inside the ambiguity band) and appends the kept processes (q', j', j'') in order to a queue,
// which the block evaluates 128 at a time, one process per thread.  With adaptive broadening the
// width of a process comes from v' - v'' (prefiltered in FP32 the same way, exact FP64 otherwise).
//
// Bound: the FP64 pipe (64 FP32 operations per FP64 one on this GPU).  A process costs
// 9 n_keys + 12 groups complex multiply-adds (354 for the diamond cell; cluster by cluster it took
// 1274), and the queue keeps the warps full although only 1-2 % of the candidates are kept.  All modes
// of a 12^3 mesh (2 x 9.5e6 processes): 71.8 ms, against 359 ms for one block per mode that evaluated
// the ~11 processes of every (128 q', j') at a time; one q point of 6^3: 0.1 against 2.0 ms a channel.
#include "fc4_window.cuh"

namespace fc4 {

constexpr int kR3Threads = 128;
// Partner points per block.  The span is a constant, so that the partial sums, and with them the
// bits of Γ, do not depend on how many modes a call or a chunk holds.
constexpr int kSpan3 = 128;

// partner branches j' tested per compaction (bounds the queue: kR3Threads * jb3 * nb entries)
constexpr int jb3(int nb) { return nb <= 6 ? nb : nb <= 12 ? 3 : 1; }

template <int NA, bool ADA>
__global__ void __launch_bounds__(kR3Threads, 4)
rates3_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch, int n_span) {
    constexpr int NB = 3 * NA, JB = jb3(NB);
    const int s = (ch == 0) ? 1 : -1;
    const double sym = (ch == 0) ? 1.0 : 0.5;
    const int N = t.N, nk = t.n_keys3;
    extern __shared__ __align__(16) unsigned char smem[];
    double2 *sG = reinterpret_cast<double2 *>(smem);            // [nk][9]
    unsigned *sList = reinterpret_cast<unsigned *>(sG + nk * 9);   // queue of kept (q' - span start, j', j'')
    __shared__ double2 se0[NB];
    __shared__ int s_scan[32];
    __shared__ double s_red[5 * 32];
    __shared__ long long s_redn[32];

    const int ms = blockIdx.x / n_span, span = blockIdx.x - ms * n_span;
    const int m0 = a.modes[ms];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    const int qlo = span * kSpan3, qhi = min(N, qlo + kSpan3);
    double acc_g = 0.0, acc_wp = 0.0;
    double acc_d[3] = {0.0, 0.0, 0.0};         // iterative BTE (a.part_d set): Σ γ Σ_k s_k ω_k F_k
    long long acc_n = 0;
    if (!(q0 == 0 && j0 < 3)) {
        const int4 c0 = t.qc[q0];
        const double w0 = t.om[m0];
        const float w0f = t.om32[m0];
        for (int k = threadIdx.x; k < NB; k += kR3Threads) se0[k] = t.ev[(q0 * NB + k) * NB + j0];
        __syncthreads();
        for (int k = threadIdx.x; k < nk * 9; k += kR3Threads) {
            const int r = k / 9, bg = k - 9 * r;
            double2 g = czero<double2>();
            for (int i = t.k3_start[r]; i < t.k3_start[r + 1]; ++i) {
                const int c = t.k3_idx[i], a0 = t.c3_at[c].x;
                const double *phi = t.phi3 + 27 * c + bg;
                double2 v = czero<double2>();
#pragma unroll
                for (int al = 0; al < 3; ++al) v = crfma(phi[9 * al], se0[3 * a0 + al], v);
                const double2 ph = cconj(t.rt[phase_index(c0, t.c3_r2[c], t.L)]);
                g = cfma(cmake(ph.x * t.c3_ism[c], ph.y * t.c3_ism[c]), v, g);
            }
            sG[k] = g;
        }
        // one process per thread: entries [first, first + 128) of the queue
        auto evaluate = [&](int it) {
            const unsigned e = sList[it];
            const int iq1 = qlo + (int)(e >> 16), j1 = (int)((e >> 8) & 0xff), j2 = (int)(e & 0xff);
            const int4 cc1 = t.qc[iq1];
            const int iq2 = q_index(c0.x + s * cc1.x, c0.y + s * cc1.y, c0.z + s * cc1.z,
                                    t.mesh[0], t.mesh[1], t.mesh[2]);
            const int m1 = iq1 * NB + j1, m2 = iq2 * NB + j2;
            const double2 *P = t.P3 + (size_t)iq1 * nk;
            const double2 *e1p = t.ev + (size_t)iq1 * NB * NB + j1, *e2p = t.ev + (size_t)iq2 * NB * NB + j2;
            double2 V = czero<double2>();
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
                        const double2 ph = cconj_if(P[r], s < 0);
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
                        V = cfma(cconj_if(e1p[(3 * b + be) * NB], s < 0), u, V);
                    }
                }
            const double d = delta_exact(ch, w0, t.om[m1], t.om[m2], 0.0);
            double g;
            if constexpr (ADA) g = gauss_adaptive(t, a, d, m1, m2);
            else g = exp(-(d * d) * a.inv_sigma2) * a.gnorm;
            const double w = sym * occupation_factor<double>(ch, t.occ[m1], t.occ[m2], 0.0) * g *
                             t.invw[m0] * t.invw[m1] * t.invw[m2];
            const double gp = w * (V.x * V.x + V.y * V.y);
            acc_wp += w;
            acc_g += gp;
            acc_n += 1;
            if (a.part_d) {                            // partner signs: 3ph+ (-, +), 3ph- (+, +)
                const double o1 = (ch == 0 ? -1.0 : 1.0) * t.om[m1], o2 = t.om[m2];
#pragma unroll
                for (int x = 0; x < 3; ++x)
                    acc_d[x] += gp * (o1 * a.bte_F[3 * m1 + x] + o2 * a.bte_F[3 * m2 + x]);
            }
        };
        int queued = 0;
        for (int qb = qlo; qb < qhi; qb += kR3Threads) {
            const int q1 = qb + threadIdx.x;
            int q2 = 0;
            unsigned v1 = 0, v2 = 0;
            if (q1 < qhi) {
                const int4 c1 = t.qc[q1];
                q2 = q_index(c0.x + s * c1.x, c0.y + s * c1.y, c0.z + s * c1.z, t.mesh[0], t.mesh[1], t.mesh[2]);
                v1 = t.vmask[q1];
                v2 = t.vmask[q2];
            }
            for (int jb = 0; jb < NB; jb += JB) {
                unsigned kept[JB];
                int n = 0;
#pragma unroll
                for (int jj = 0; jj < JB; ++jj) {
                    const int j1 = jb + jj;
                    kept[jj] = 0;
                    if (!((v1 >> j1) & 1u)) continue;
                    // window: this thread's (q', j') against every j''
                    const float base32 = w0f + (float)s * t.om32[q1 * NB + j1];
                    const int m1 = q1 * NB + j1;
                    for (int j2 = 0; j2 < NB; ++j2) {
                        if (!((v2 >> j2) & 1u)) continue;
                        const int m2 = q2 * NB + j2;
                        const float ad = fabsf(base32 - t.om32[m2]);
                        bool keep;
                        if constexpr (ADA) {
                            const int w = window_adaptive32(a, ad, two_sigma32(t, a, m1, m2));
                            keep = w == 2 || (w == 1 && window_exact_adaptive(t, a, ch, m0, m1, m2, -1, m1, m2));
                        } else {
                            if (ad <= a.lo32) keep = true;
                            else if (ad > a.hi32) keep = false;
                            else keep = fabs(delta_exact(ch, w0, t.om[m1], t.om[m2], 0.0)) <= a.two_sigma;
                        }
                        kept[jj] |= (unsigned)keep << j2;
                    }
                    n += __popc(kept[jj]);
                }
                int total;
                int off = queued + block_exclusive_scan(n, s_scan, &total);     // also orders sG
#pragma unroll
                for (int jj = 0; jj < JB; ++jj) {
                    unsigned m = kept[jj];
                    while (m) {
                        const int j2 = __ffs(m) - 1;
                        m &= m - 1;
                        sList[off++] = ((unsigned)(q1 - qlo) << 16) | ((unsigned)(jb + jj) << 8) | (unsigned)j2;
                    }
                }
                queued += total;
                __syncthreads();
                if (queued >= kR3Threads) {            // full rounds from the tail; < 128 entries stay
                    for (; queued >= kR3Threads; queued -= kR3Threads)
                        evaluate(queued - kR3Threads + (int)threadIdx.x);
                    __syncthreads();                   // the tail is overwritten by the next append
                }
            }
        }
        if ((int)threadIdx.x < queued) evaluate(threadIdx.x);
    }
    double sums[5] = {acc_g, acc_wp, acc_d[0], acc_d[1], acc_d[2]};
    long long cnts[1] = {acc_n};
    block_sum_multi<5, 1>(sums, cnts, s_red, s_redn);
    if (threadIdx.x == 0) {
        const size_t o = ((size_t)ch * a.n_modes + ms) * N + span;
        if (a.part_d)
            for (int x = 0; x < 3; ++x) a.part_d[3 * o + x] = sums[2 + x] * t.invw[m0];
        a.part_g[o] = sums[0];
        a.part_wp[o] = sums[1];
        a.part_n[o] = cnts[0];
        a.part_items[o] = 0;
        a.part_ent[o] = 0;
        if (a.part_ev) a.part_ev[o] = cnts[0];
        if (a.part_cev) a.part_cev[o] = (long long)(qhi - qlo) * NB * NB;
    }
}

template <int NA>
static cudaError_t launch3(const Tables &t, RateArgs &a, int ch, cudaStream_t s) {
    constexpr int NB = 3 * NA;
    const int n_span = (t.N + kSpan3 - 1) / kSpan3;
    a.n_part[ch] = n_span;
    if (a.n_modes == 0) return cudaSuccess;
    const size_t smem = sizeof(double2) * (size_t)t.n_keys3 * 9 +
                        sizeof(unsigned) * (size_t)kR3Threads * (jb3(NB) * NB + 1);
    if ((long long)a.n_modes * n_span > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    auto kern = a.adaptive ? rates3_kernel<NA, true> : rates3_kernel<NA, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((long long)a.n_modes * n_span), kR3Threads, smem, s>>>(t, a, ch, n_span);
    e = cudaGetLastError();
    if (e == cudaSuccess && a.n_kernels) ++*a.n_kernels;
    return e;
}

cudaError_t launch_rates3(const Tables &t, RateArgs &a, int ch, int fp64, cudaStream_t s) {
    (void)fp64;
    switch (t.n_atoms) {
    case 1: return launch3<1>(t, a, ch, s);
    case 2: return launch3<2>(t, a, ch, s);
    case 3: return launch3<3>(t, a, ch, s);
    case 4: return launch3<4>(t, a, ch, s);
    case 5: return launch3<5>(t, a, ch, s);
    case 6: return launch3<6>(t, a, ch, s);
    case 7: return launch3<7>(t, a, ch, s);
    case 8: return launch3<8>(t, a, ch, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fc4
