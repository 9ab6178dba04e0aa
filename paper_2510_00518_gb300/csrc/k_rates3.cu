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
// Bound: the FP64 pipe (64 FP32 operations per FP64 one on this GPU); cluster by cluster a process took
// 1274 complex multiply-adds.  Cells of up to two atoms (rates3_pair_kernel) list the points (λ, q') with a
// kept process, form T[bβ][cγ] = Σ_r P_r G_r[βγ] once per point (198 for the diamond cell,
// mirror keys paired) and take the
// 2-3 processes of a point at 42 each, on full warps.  Larger cells (rates3_kernel) evaluate a process
// per thread at 9 n_keys + 12 groups each (their T does not fit in registers).  3ph- is evaluated on half of
// its pairs where Φ3 allows it, and both channels share a launch.  All modes of 12^3 (2 x 9.5e6
// processes): 359 ms for one block per mode and ~11 processes at a time, 70 ms with a process per thread
// and 28 ms so, 23.5 with mirror keys paired; eight atoms, one q of 4^3: 55, 13 and 1.7 ms.
#include "k_rates3.cuh"

namespace fc4 {

// Partner points per block.  The span depends on the cell alone, so that the partial sums, and with them
// the bits of Γ, do not depend on how many modes a call or a chunk holds.  512 points hold ~100 active
// ones of a two-atom cell (a few warps' worth); a point of a larger cell carries nb^2 branch pairs, and
// ~128 processes per block keep small calls spread over the SMs.
constexpr int kSpan3Pair = 512;
constexpr int span3(int nb) { return 4608 / (nb * nb) < 8 ? 8 : 4608 / (nb * nb); }

// Channel of a block: launches over both channels have them in grid dimension y.
__device__ __forceinline__ int channel3(int mask) { return mask == 3 ? (int)blockIdx.y : mask - 1; }

template <int NA, bool ADA>
__global__ void __launch_bounds__(kR3Threads, 2)
rates3_pair_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int mask, int n_span) {
    constexpr int NB = 3 * NA;
    using C = double2;
    const int N = t.N, nk = t.n_keys3;
    extern __shared__ __align__(16) unsigned char smem[];
    C *sG = reinterpret_cast<C *>(smem);                        // [nk][9], in the FP64 key order
    __shared__ unsigned long long s_list[kSpan3Pair];           // points: q' - qlo, domain code, kept (j', j'')
    __shared__ unsigned short s_proc[kR3Threads * NB * NB];     // per warp: processes (lane, j', j'') of 32 points
    __shared__ C se0[NB];
    __shared__ int s_scan[32];
    __shared__ double s_red[5 * 32];
    __shared__ long long s_redn[3 * 32];

    const int ch = channel3(mask);
    const int ms = blockIdx.x / n_span, span = blockIdx.x - ms * n_span;
    const int qlo = span * kSpan3Pair, qhi = min(N, qlo + kSpan3Pair);
    const Three p(t, ch, a.modes[ms], NB);
    // 3ph- is symmetric under (λ', λ'') (q' <-> q'' = q - q'): one process of each swapped pair, weight 2
    const bool tri = ch == 1 && (a.tri & *t.domains & 4);
    double acc_g = 0.0, acc_wp = 0.0;
    double acc_d[3] = {0.0, 0.0, 0.0};         // iterative BTE (a.part_d set): Σ γ Σ_k s_k ω_k F_k
    long long acc_n = 0, acc_ev = 0, acc_cev = 0;
    if (!(p.q0 == 0 && p.j0 < 3)) {
        for (int k = threadIdx.x; k < NB; k += kR3Threads) se0[k] = t.ev[(p.q0 * NB + k) * NB + p.j0];
        __syncthreads();
        three_G<true>(t, p, se0, sG);
        __syncthreads();
        for (int k = threadIdx.x; k < nk * 9; k += kR3Threads)     // mirror pairs x, y -> x + y, i (x - y) in place;
            if (t.perm3[k / 9] >> 28 == 1) {                       // ordered before its use by the scans' barriers
                const C x = sG[k], y = sG[k + 9];
                sG[k] = cmake(x.x + y.x, x.y + y.y);
                sG[k + 9] = cmake(y.y - x.y, x.x - y.x);
            }
        int total = 0;
        for (int qb = qlo; qb < qhi; qb += kR3Threads) {
            const int q1 = qb + threadIdx.x;
            unsigned long long kept = 0;
            int code = 0;                      // 0: weight 1; 1: weight 2; 2: q' = q''
            if (q1 < qhi) {
                const int4 c1 = t.qc[q1];
                const int q2 = q_index(p.c0.x + p.s * c1.x, p.c0.y + p.s * c1.y, p.c0.z + p.s * c1.z,
                                       t.mesh[0], t.mesh[1], t.mesh[2]);
                if (!tri || q1 <= q2) {
                    code = !tri ? 0 : q1 < q2 ? 1 : 2;
                    acc_cev += NB * NB;
                    const unsigned v1 = t.vmask[q1], v2 = t.vmask[q2];
                    float w2[NB];
#pragma unroll
                    for (int j2 = 0; j2 < NB; ++j2) w2[j2] = t.om32[q2 * NB + j2];
#pragma unroll
                    for (int j1 = 0; j1 < NB; ++j1) {
                        if (!((v1 >> j1) & 1u)) continue;
                        const int m1 = q1 * NB + j1;
                        const float base32 = p.w0f + (float)p.s * t.om32[m1];
                        unsigned near = 0;
                        if constexpr (ADA) near = v2;
                        else {
#pragma unroll
                            for (int j2 = 0; j2 < NB; ++j2) near |= (unsigned)(fabsf(base32 - w2[j2]) <= a.hi32) << j2;
                            near &= v2;
                        }
                        if (code == 2) near &= ~((1u << j1) - 1u);            // j'' >= j'
                        for (; near; near &= near - 1) {
                            const int j2 = __ffs(near) - 1, m2 = q2 * NB + j2;
                            const float ad = fabsf(base32 - t.om32[m2]);
                            bool keep;
                            if constexpr (ADA) {
                                const int w = window_adaptive32(a, ad, two_sigma32(t, a, m1, m2));
                                keep = w == 2 || (w == 1 && window_exact_adaptive(t, a, ch, p.m0, m1, m2, -1, m1, m2));
                            } else {
                                keep = ad <= a.lo32 || fabs(delta_exact(ch, p.w0, t.om[m1], t.om[m2], 0.0)) <= a.two_sigma;
                            }
                            kept |= (unsigned long long)keep << (NB * j1 + j2);
                        }
                    }
                }
            }
            int n;
            const int o = block_exclusive_scan(kept != 0, s_scan, &n);
            if (kept) s_list[total + o] = ((unsigned long long)(q1 - qlo) << 48) | ((unsigned long long)code << 40) | kept;
            total += n;
        }
        __syncthreads();
        // 32 points to a warp: a lane forms its point's T, and the processes of the 32 points go one to a lane.
        // The first warp differs from mode to mode (each has its own scheduler's FP64 pipe) but not from block to
        // block: the order of the sums must not depend on the chunk or the subset.
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        unsigned short *wProc = s_proc + wid * 32 * NB * NB;
        for (int pb = ((wid + p.m0 + span) & 3) * 32; pb < total; pb += kR3Threads) {
            unsigned long long e = 0;
            int iq1 = 0, iq2 = 0;
            C T[NA][NA][9];
            if (pb + lane < total) {
                e = s_list[pb + lane];
                iq1 = qlo + (int)(e >> 48);
                const int4 cc1 = t.qc[iq1];
                iq2 = q_index(p.c0.x + p.s * cc1.x, p.c0.y + p.s * cc1.y, p.c0.z + p.s * cc1.z,
                              t.mesh[0], t.mesh[1], t.mesh[2]);
                const C *P = t.P3 + (size_t)iq1 * nk;
#pragma unroll
                for (int b = 0; b < NA; ++b)
#pragma unroll
                    for (int c = 0; c < NA; ++c)
                        paired_sum(t.perm3, t.grp3_start[b * NA + c], t.pairs3[b * NA + c], t.grp3_start[b * NA + c + 1], P, sG,
                                   (double)p.s, T[b][c]);
            }
            const unsigned long long kept = e & ((1ull << (NB * NB)) - 1ull);
            const int np = __popcll(kept);
            int o = warp_exclusive_scan(np);
            const int n_proc = __shfl_sync(kFull, o + np, 31);
            for (unsigned long long m = kept; m; m &= m - 1) wProc[o++] = (unsigned short)((lane << 6) | (__ffsll(m) - 1));
            __syncwarp();
            for (int pp = 0; pp < n_proc; pp += 32) {
                const bool act = pp + lane < n_proc;
                const int pc = act ? wProc[pp + lane] : 0;
                const int src = pc >> 6, j1 = (pc & 63) / NB, j2 = (pc & 63) % NB;
                const int sq1 = __shfl_sync(kFull, iq1, src), sq2 = __shfl_sync(kFull, iq2, src);
                const int code = (int)(__shfl_sync(kFull, e, src) >> 40) & 3;
                const int m1 = sq1 * NB + j1, m2 = sq2 * NB + j2;
                const C *e1p = t.ev + (size_t)sq1 * NB * NB + j1, *e2p = t.ev + (size_t)sq2 * NB * NB + j2;
                C e2[NB], V = czero<C>();
#pragma unroll
                for (int k = 0; k < NB; ++k) e2[k] = cconj(e2p[k * NB]);
#pragma unroll
                for (int b = 0; b < NA; ++b)
#pragma unroll
                    for (int be = 0; be < 3; ++be) {
                        C u = czero<C>();
#pragma unroll
                        for (int k = 0; k < NB; ++k) u = cfma(cshfl(T[b][k / 3][3 * be + k % 3], src), e2[k], u);
                        V = cfma(cconj_if(e1p[(3 * b + be) * NB], p.s < 0), u, V);
                    }
                const double d = delta_exact(ch, p.w0, t.om[m1], t.om[m2], 0.0);
                double g;
                if constexpr (ADA) g = gauss_adaptive(t, a, d, m1, m2);
                else g = exp(-(d * d) * a.inv_sigma2) * a.gnorm;
                const int wt = code == 0 ? 1 : code == 1 ? 2 : j1 < j2 ? 2 : 1;
                const double w = wt * (ch == 0 ? 1.0 : 0.5) * occupation_factor<double>(ch, t.occ[m1], t.occ[m2], 0.0) * g *
                                 t.invw[p.m0] * t.invw[m1] * t.invw[m2];
                if (act) {
                    const double gp = w * (V.x * V.x + V.y * V.y);
                    acc_wp += w;
                    acc_g += gp;
                    acc_n += wt;
                    acc_ev += 1;
                    if (a.part_d) {                    // partner signs: 3ph+ (-, +), 3ph- (+, +)
                        const double o1 = (ch == 0 ? -1.0 : 1.0) * t.om[m1], o2 = t.om[m2];
#pragma unroll
                        for (int x = 0; x < 3; ++x)
                            acc_d[x] += gp * (o1 * a.bte_F[3 * m1 + x] + o2 * a.bte_F[3 * m2 + x]);
                    }
                }
            }
            __syncwarp();                                        // wProc reused
        }
    }
    double sums[5] = {acc_g, acc_wp, acc_d[0], acc_d[1], acc_d[2]};
    long long cnts[3] = {acc_n, acc_ev, acc_cev};
    block_sum_multi<5, 3>(sums, cnts, s_red, s_redn);
    if (threadIdx.x == 0) {
        const size_t o = ((size_t)ch * a.n_modes + ms) * N + span;
        if (a.part_d)
            for (int x = 0; x < 3; ++x) a.part_d[3 * o + x] = sums[2 + x] * t.invw[p.m0];
        a.part_g[o] = sums[0];
        a.part_wp[o] = sums[1];
        a.part_n[o] = cnts[0];
        a.part_items[o] = 0;
        a.part_ent[o] = 0;
        if (a.part_ev) a.part_ev[o] = cnts[1];
        if (a.part_cev) a.part_cev[o] = cnts[2];
    }
}

template <int NA, bool ADA, int JB>
__global__ void __launch_bounds__(kR3Threads, 4)
rates3_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int mask, int n_span) {
    constexpr int NB = 3 * NA, kSpan3 = span3(NB);
    static_assert(kSpan3 <= kQueueSpan3, "a queued process holds q' - qlo in 16 bits");
    const int ch = channel3(mask);
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
        three_G<false>(t, p, se0, sG);         // ordered before its use by the first append's barriers
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
                queued = three_append<NB, ADA, JB>(t, a, p, qlo, qb, qhi, jb, queued, sList, s_scan);
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

// The pair kernel serves cells of up to two atoms whose G fits beside its lists (1500 keys); larger lists, and larger
// cells, take rates3_kernel, with one partner branch a round (a shorter queue) where the G of the usual rounds would
// not fit (1567 keys for two atoms, 1499 for eight).  Clusters with a key each, two atoms, one q of 5^3, σ 2 THz,
// cluster by cluster and now: 900 clusters 62.9 and 1.4 ms, 1540 clusters 115.6 and 2.2 ms.
template <int NA>
static cudaError_t launch3(const Tables &t, RateArgs &a, int mask, cudaStream_t s) {
    constexpr int NB = 3 * NA, JB = jb3(NB);
    constexpr size_t kMost = 227 * 1024, kPairStatic = 16 * 1024, kStatic = 3 * 1024;   // with static shared memory
    const size_t g = sizeof(double2) * 9 * (size_t)t.n_keys3;
    auto queue = [](int jb) { return sizeof(unsigned) * (size_t)kR3Threads * (jb * NB + 1); };
    const bool few = NA <= 2 && g + kPairStatic <= kMost;
    const int jb = NA <= 2 || g + queue(JB) + kStatic > kMost ? 1 : JB;
    const int per = few ? kSpan3Pair : span3(NB), n_span = (t.N + per - 1) / per;
    for (int ch = 0; ch < 2; ++ch)
        if ((mask >> ch) & 1) a.n_part[ch] = n_span;
    if (a.n_modes == 0 || !mask) return cudaSuccess;
    const size_t smem = few ? g : g + queue(jb);
    if ((long long)a.n_modes * n_span > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    void (*kern)(Tables, RateArgs, int, int) = a.adaptive ? rates3_kernel<NA, true, 1> : rates3_kernel<NA, false, 1>;
    if constexpr (NA <= 2) {
        if (few) kern = a.adaptive ? rates3_pair_kernel<NA, true> : rates3_pair_kernel<NA, false>;
    } else if (jb != 1) {
        kern = a.adaptive ? rates3_kernel<NA, true, JB> : rates3_kernel<NA, false, JB>;
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3((unsigned)((long long)a.n_modes * n_span), mask == 3 ? 2 : 1), kR3Threads, smem, s>>>(t, a, mask, n_span);
    e = cudaGetLastError();
    if (e == cudaSuccess && a.n_kernels) ++*a.n_kernels;
    return e;
}

cudaError_t launch_rates3(const Tables &t, RateArgs &a, int mask, cudaStream_t s) {
    switch (t.n_atoms) {
    case 1: return launch3<1>(t, a, mask, s);
    case 2: return launch3<2>(t, a, mask, s);
    case 3: return launch3<3>(t, a, mask, s);
    case 4: return launch3<4>(t, a, mask, s);
    case 5: return launch3<5>(t, a, mask, s);
    case 6: return launch3<6>(t, a, mask, s);
    case 7: return launch3<7>(t, a, mask, s);
    case 8: return launch3<8>(t, a, mask, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fc4
