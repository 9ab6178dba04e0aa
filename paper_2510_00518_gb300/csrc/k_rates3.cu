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
#include "k_rates3.cuh"

namespace fc4 {

// Partner points per block.  The span is a constant, so that the partial sums, and with them the
// bits of Γ, do not depend on how many modes a call or a chunk holds.
constexpr int kSpan3 = 128;

template <int NA, bool ADA>
__global__ void __launch_bounds__(kR3Threads, 4)
rates3_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch, int n_span) {
    constexpr int NB = 3 * NA, JB = jb3(NB);
    const int N = t.N;
    extern __shared__ __align__(16) unsigned char smem[];
    double2 *sG = reinterpret_cast<double2 *>(smem);            // [n_keys3][9]
    unsigned *sList = reinterpret_cast<unsigned *>(sG + t.n_keys3 * 9);   // queue of kept processes
    __shared__ double2 se0[NB];
    __shared__ int s_scan[32];
    __shared__ double s_red[5 * 32];
    __shared__ long long s_redn[32];

    const int ms = blockIdx.x / n_span, span = blockIdx.x - ms * n_span;
    const int qlo = span * kSpan3, qhi = min(N, qlo + kSpan3);
    const Three p(t, ch, a.modes[ms], NB);
    double acc_g = 0.0, acc_wp = 0.0;
    double acc_d[3] = {0.0, 0.0, 0.0};         // iterative BTE (a.part_d set): Σ γ Σ_k s_k ω_k F_k
    long long acc_n = 0;
    if (!(p.q0 == 0 && p.j0 < 3)) {
        for (int k = threadIdx.x; k < NB; k += kR3Threads) se0[k] = t.ev[(p.q0 * NB + k) * NB + p.j0];
        __syncthreads();
        three_G(t, p, se0, sG);                // ordered before its use by the first append's barriers
        auto evaluate = [&](int it) {
            const ThreeProcess z = three_evaluate<NA, ADA>(t, a, p, qlo, sList[it], sG);
            const double gp = z.w * (z.V.x * z.V.x + z.V.y * z.V.y);
            acc_wp += z.w;
            acc_g += gp;
            acc_n += 1;
            if (a.part_d) {                            // partner signs: 3ph+ (-, +), 3ph- (+, +)
                const double o1 = (ch == 0 ? -1.0 : 1.0) * t.om[z.m1], o2 = t.om[z.m2];
#pragma unroll
                for (int x = 0; x < 3; ++x)
                    acc_d[x] += gp * (o1 * a.bte_F[3 * z.m1 + x] + o2 * a.bte_F[3 * z.m2 + x]);
            }
        };
        int queued = 0;
        for (int qb = qlo; qb < qhi; qb += kR3Threads)
            for (int jb = 0; jb < NB; jb += JB) {
                queued = three_append<NB, ADA>(t, a, p, qlo, qb, qhi, jb, queued, sList, s_scan);
                if (queued >= kR3Threads) {            // full rounds from the tail; < 128 entries stay
                    for (; queued >= kR3Threads; queued -= kR3Threads)
                        evaluate(queued - kR3Threads + (int)threadIdx.x);
                    __syncthreads();                   // the tail is overwritten by the next append
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
            for (int x = 0; x < 3; ++x) a.part_d[3 * o + x] = sums[2 + x] * t.invw[p.m0];
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
