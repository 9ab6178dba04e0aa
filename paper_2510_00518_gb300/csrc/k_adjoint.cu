// k_adjoint.cu - adjoint of the scattering rates with respect to the cubic and quartic force
// constants, at fixed modes and fixed σ, FP64, deterministic.
//
// L = Σ_{ch,λ} dL/dΓ_ch(λ) Γ_ch(λ) and Γ = C/N^k Σ_p w_p |V_p|², so with G_p = dL/dΓ(λ) C/N^k w_p
//   dL/dΦ_c[..] = Σ_p G_p 2 Re(conj(V_p) dV_p/dΦ_c[..]),   dV_p/dΦ_c = phase_c e e e (e) / sqrt(m),
// and V is recomputed (never stored).
//
// Four-phonon: one block per mode λ loops over (q', j').  With W_r, P_r and the keys of the forward
// kernel, V = Σ_r P_r^s2 Σ_γδ W_r[γδ] e^s2''(cγ) e*'''(dδ), and the gradient factorises through
//   Ȳ[cγ] = Σ_j'' G conj(V) e^s2''(cγ)          (per (q'', j''') item)
//   H_r[γδ] = Σ_items P_r^s2 Ȳ[c_r γ] e*'''(d_r δ) (per (λ, q', j'), owner threads, fixed order)
//   dL/dΦ_c[αβγδ] += 2 Re(phase_c / sqrt(m) e_λ(aα) e^s1'(bβ) H_{r(c)}[γδ]).
// Items of each q'' round are compacted into shared memory one per thread at a time, and every
// H entry is summed by the thread that owns it, in item order.  Each block writes its gradient
// into its own slice; a final kernel sums the slices over λ in order.
#include "k_rates3.cuh"
#include "k_rates4_tile.cuh"

namespace fc4 {

constexpr int kAdjThreads = 128;

// Kahan-compensated FP32 accumulation in a (sum, compensation) pair (mixed-precision slices)
__device__ __forceinline__ void kahan_add(float2 &acc, float x) {
    const float y = x - acc.y;
    const float t = acc.x + y;
    acc.y = (t - acc.x) - y;
    acc.x = t;
}

// ------------------------------------------------------------------------------ four-phonon

template <typename R, int NA>
struct Item4 {
    int q2, q3;
    Cplx<R> ybar[3 * NA];
    Cplx<R> e3c[3 * NA];
};

template <typename R, int NA>
__global__ void __launch_bounds__(kAdjThreads)
adj4_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch,
            const double *__restrict__ dLdG, double cst, double *dphi_part) {
    constexpr int NB = 3 * NA;
    using C = Cplx<R>;
    const C *ev = Sel<R>::ev(t);
    const C *rt = Sel<R>::rt(t);
    const C *P4 = Sel<R>::P4(t);
    const R *phi4 = Sel<R>::phi4(t);
    const R *ism4 = Sel<R>::ism4(t);
    const int s1 = (ch == 4) ? -1 : 1;
    const int s2 = (ch == 2) ? 1 : -1;
    const int N = t.N, nk = t.n_keys, nc4 = t.nc4;
    extern __shared__ __align__(16) unsigned char smem[];
    C *sW = reinterpret_cast<C *>(smem);                        // [nk][9]
    C *sH = sW + nk * 9;                                        // [nk][9]
    C *sCon = sH + nk * 9;                                      // [nc4][9] per-cluster terms of W
    C *sPh = sCon + nc4 * 9;                                    // [nc4] phase / sqrt(m) at (q, q')
    C *sE = sPh + nc4;                                          // [NA*NA][9]
    C *se0 = sE + NA * NA * 9;                                  // [NB]
    Item4<R, NA> *sIt = reinterpret_cast<Item4<R, NA> *>(se0 + NB);   // [kAdjThreads]
    __shared__ int s_scan[32];
    __shared__ int s_max;

    const int ms = blockIdx.x;
    const int m0 = a.modes[ms];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    // per-mode gradient slice: FP64, or (mixed) FP32 Kahan pairs (sum, compensation) in the same bytes
    double *dphi = dphi_part + (size_t)ms * nc4 * 81;
    float2 *dphk = reinterpret_cast<float2 *>(dphi);
    for (int k = threadIdx.x; k < nc4 * 81; k += kAdjThreads) {
        if constexpr (sizeof(R) == 8) dphi[k] = 0.0;
        else dphk[k] = make_float2(0.0f, 0.0f);
    }
    const double gl = dLdG[(size_t)ch * a.n_modes + ms] * cst;
    if ((q0 == 0 && j0 < 3) || gl == 0.0) return;
    const int4 c0 = t.qc[q0];
    const double w0 = t.om[m0];
    const float w0f = t.om32[m0];
    for (int k = threadIdx.x; k < NB; k += kAdjThreads) se0[k] = ev[(q0 * NB + k) * NB + j0];

    for (int q1 = 0; q1 < N; ++q1) {
        const int4 c1 = t.qc[q1];
        const int b0 = c0.x + s1 * c1.x, b1 = c0.y + s1 * c1.y, b2 = c0.z + s1 * c1.z;
        const unsigned vm1 = t.vmask[q1];
        for (int j1 = 0; j1 < NB; ++j1) {
            if (!((vm1 >> j1) & 1u)) continue;
            const int m1 = q1 * NB + j1;
            const double w1 = t.om[m1];
            __syncthreads();
            for (int k = threadIdx.x; k < NA * NA * 9; k += kAdjThreads) {
                const int ab = k / 9, ij = k - ab * 9;
                const int at = ab / NA, bt = ab - at * NA;
                const int al = ij / 3, be = ij - al * 3;
                sE[k] = cmul(se0[3 * at + al], cconj_if(ev[(q1 * NB + 3 * bt + be) * NB + j1], s1 < 0));
            }
            for (int c = threadIdx.x; c < nc4; c += kAdjThreads) {
                const C p = rt[mod_pos(s1 * phase_index(c1, t.c4_r13[c], t.L) - phase_index(c0, t.c4_r3[c], t.L), t.L)];
                sPh[c] = cmake(p.x * ism4[c], p.y * ism4[c]);
            }
            for (int k = threadIdx.x; k < nk * 9; k += kAdjThreads) sH[k] = czero<C>();
            __syncthreads();
            for (int k = threadIdx.x; k < nc4 * 9; k += kAdjThreads) {
                const int c = k / 9, gd = k - c * 9;
                const int4 at = t.c4_at[c];
                const R *ph4 = phi4 + 81 * c + gd;
                const C *E = sE + (at.x * NA + at.y) * 9;
                C v = czero<C>();
#pragma unroll
                for (int ab = 0; ab < 9; ++ab) v = crfma(ph4[9 * ab], E[ab], v);
                sCon[k] = cmul(sPh[c], v);
            }
            __syncthreads();
            for (int k = threadIdx.x; k < nk * 9; k += kAdjThreads) {
                const int r = k / 9, gd = k - r * 9;
                C acc = czero<C>();
                for (int c = t.key_start[r]; c < t.key_start[r + 1]; ++c) acc = cadd(acc, sCon[c * 9 + gd]);
                sW[k] = acc;
            }
            __syncthreads();
            const float base32 = w0f + (float)s1 * t.om32[m1];
            for (int qb = 0; qb < N; qb += kAdjThreads) {
                const int q2 = qb + threadIdx.x;
                unsigned mask[NB];
                int q3 = 0, n_it = 0;
                if (q2 < N) {
                    const int4 c2 = t.qc[q2];
                    q3 = q_index(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z, t.mesh[0], t.mesh[1], t.mesh[2]);
                    const unsigned v2 = t.vmask[q2], v3 = t.vmask[q3];
                    for (int j3 = 0; j3 < NB; ++j3) {
                        unsigned m = 0;
                        if ((v3 >> j3) & 1u)
                            for (int j2 = 0; j2 < NB; ++j2) {
                                if (!((v2 >> j2) & 1u)) continue;
                                const float ad = fabsf((base32 + (float)s2 * t.om32[q2 * NB + j2]) - t.om32[q3 * NB + j3]);
                                bool keep;
                                if (a.adaptive) {
                                    const int mm2 = q2 * NB + j2, mm3 = q3 * NB + j3;
                                    const int w = window_adaptive32(a, ad, two_sigma32(t, a, mm2, mm3));
                                    keep = w == 2 || (w == 1 && window_exact_adaptive(t, a, ch, m0, m1, mm2, mm3, mm2, mm3));
                                } else if (ad <= a.lo32) keep = true;
                                else if (ad > a.hi32) keep = false;
                                else keep = fabs(delta_exact(ch, w0, w1, t.om[q2 * NB + j2], t.om[q3 * NB + j3])) <= a.two_sigma;
                                m |= (unsigned)keep << j2;
                            }
                        mask[j3] = m;
                        n_it += (m != 0);
                    }
                } else {
                    for (int j3 = 0; j3 < NB; ++j3) mask[j3] = 0;
                }
                if (threadIdx.x == 0) s_max = 0;
                __syncthreads();
                atomicMax(&s_max, n_it);
                __syncthreads();
                const int rounds = s_max;
                int next_j3 = 0;
                for (int sr = 0; sr < rounds; ++sr) {
                    // this thread's next item (q'', j''')
                    int j3 = -1;
                    while (next_j3 < NB && j3 < 0) {
                        if (mask[next_j3]) j3 = next_j3;
                        ++next_j3;
                    }
                    Item4<R, NA> it;
                    if (j3 >= 0) {
                        C Y[NA][3];
                        for (int c = 0; c < NA; ++c)
                            for (int g = 0; g < 3; ++g) Y[c][g] = czero<C>();
                        const C *P = P4 + (size_t)q2 * nk;
                        for (int c = 0; c < NA; ++c)
                            for (int d = 0; d < NA; ++d) {
                                C e3[3];
                                for (int dl = 0; dl < 3; ++dl) e3[dl] = cconj(ev[(q3 * NB + 3 * d + dl) * NB + j3]);
                                for (int r = t.grp_start[c * NA + d]; r < t.grp_start[c * NA + d + 1]; ++r) {
                                    const C ph = cconj_if(P[r], s2 < 0);
                                    const C *Wr = sW + 9 * r;
                                    for (int g = 0; g < 3; ++g) {
                                        C u = cmul(Wr[3 * g], e3[0]);
                                        u = cfma(Wr[3 * g + 1], e3[1], u);
                                        u = cfma(Wr[3 * g + 2], e3[2], u);
                                        Y[c][g] = cfma(ph, u, Y[c][g]);
                                    }
                                }
                            }
                        for (int k = 0; k < NB; ++k) it.ybar[k] = czero<C>();
                        const int m3 = q3 * NB + j3;
                        unsigned m = mask[j3];
                        while (m) {
                            const int j2 = __ffs(m) - 1;
                            m &= m - 1;
                            const int m2 = q2 * NB + j2;
                            C e2[NB];
                            for (int k = 0; k < NB; ++k) e2[k] = cconj_if(ev[(q2 * NB + k) * NB + j2], s2 < 0);
                            C V = czero<C>();
                            for (int c = 0; c < NA; ++c)
                                for (int g = 0; g < 3; ++g) V = cfma(e2[3 * c + g], Y[c][g], V);
                            const double d = delta_exact(ch, w0, w1, t.om[m2], t.om[m3]);
                            const double gs = a.adaptive ? gauss_adaptive(t, a, d, m2, m3)
                                                         : exp(-(d * d) * a.inv_sigma2) * a.gnorm;
                            const double w = (ch == 4 ? 1.0 / 6.0 : 0.5) *
                                             occupation_factor<double>(ch, t.occ[m1], t.occ[m2], t.occ[m3]) * gs *
                                             t.invw[m0] * t.invw[m1] * t.invw[m2] * t.invw[m3];
                            const C f = cmake((R)(gl * w * (double)V.x), (R)(-gl * w * (double)V.y));      // G conj(V)
                            for (int k = 0; k < NB; ++k) it.ybar[k] = cfma(f, e2[k], it.ybar[k]);
                        }
                        it.q2 = q2;
                        it.q3 = q3;
                        for (int k = 0; k < NB; ++k) it.e3c[k] = cconj(ev[(q3 * NB + k) * NB + j3]);
                    }
                    int total;
                    const int off = block_exclusive_scan(j3 >= 0 ? 1 : 0, s_scan, &total);
                    if (j3 >= 0) sIt[off] = it;
                    __syncthreads();
                    // owners accumulate H_r[γδ] += P_r^s2 Ȳ[c_r γ] e*'''(d_r δ) over the items, in order
                    for (int k = threadIdx.x; k < nk * 9; k += kAdjThreads) {
                        const int r = k / 9, gd = k - r * 9, g = gd / 3, dl = gd - 3 * g;
                        int grp = 0;
                        while (t.grp_start[grp + 1] <= r) ++grp;
                        const int cc = grp / NA, dd = grp - cc * NA;
                        C h = sH[k];
                        for (int i = 0; i < total; ++i) {
                            const C ph = cconj_if(P4[(size_t)sIt[i].q2 * nk + r], s2 < 0);
                            h = cfma(cmul(ph, sIt[i].ybar[3 * cc + g]), sIt[i].e3c[3 * dd + dl], h);
                        }
                        sH[k] = h;
                    }
                    __syncthreads();
                }
            }
            // fold H into the gradient: dΦ_c[αβγδ] += 2 Re(phase_c/sqrt(m) E[a,b][αβ] H_{r(c)}[γδ])
            __syncthreads();
            for (int r = 0; r < nk; ++r)
                for (int c = t.key_start[r]; c < t.key_start[r + 1]; ++c) {
                    const int4 at = t.c4_at[c];
                    for (int k = threadIdx.x; k < 81; k += kAdjThreads) {
                        const int ab = k / 9, gd = k - ab * 9;
                        const C z = cmul(cmul(sPh[c], sE[(at.x * NA + at.y) * 9 + ab]), sH[r * 9 + gd]);
                        if constexpr (sizeof(R) == 8) dphi[(size_t)c * 81 + k] += 2.0 * z.x;
                        else kahan_add(dphk[(size_t)c * 81 + k], 2.0f * z.x);
                    }
                }
        }
    }
}

// ---- FP64, cells of up to two atoms: three kernels over units (λ, q'), as the rates take them.
//
// w4_kernel leaves W[j'][r][γδ] of every unit in the W buffer.  adj4_tile_kernel owns a unit: it lists
// the entries (q'', j', kept pairs) of its window, j' by j', and takes them 128 at a time, one per thread:
// X from W, and per item and process V, Ȳ[cγ] = Σ_j'' G conj(V) e^s2_λ'' and Z[cγ,dδ] += Ȳ[cγ] e*_λ'''(dδ)
// in the thread's column of shared memory; then the owner of each (r, γδ) adds P_r^s2 Z over the
// entries of a j' into the unit's H[j'][r][γδ], which replaces its W unless there is room for both
// (++ and +- then share W: 4.4 of 92 ms).  adj4_fold_kernel owns a
// mode: per q' it forms K_rb[βγδ] = Σ_j' e^s1_λ'(bβ) H_r[j'][γδ] once for all clusters and adds
// phase_c K_r(c)b(c) to 27 numbers a cluster in registers, and expands them by e_λ(aα) into the mode's
// gradient slice at the end.
//
// Bound: FP64.  Per entry 396 + 72 items complex multiply-adds (mirror keys paired), per (λ, q') 17000 for the fold (the
// block-per-mode kernel above takes 1020 an item and 220000 a (λ, q')).  Where Φ4 has the leg-exchange
// symmetry only one process of each swapped pair is evaluated (self-swapped ones with weight 1/2) and
// sum_slices_kernel adds the gradient of the swapped legs.  κ and its gradient for all modes of a 4^3
// mesh: 634 ms with the block-per-mode kernels for both orders, 121 ms with these as first built, 95 ms with
// mirror keys paired, lanes taking their own items and the shared W.
constexpr int kAdjLd = kAdjThreads + 1;

template <int NA, bool ADA>
__global__ void __launch_bounds__(kAdjThreads, 2)
adj4_tile_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch, int mode0,
                 const double *__restrict__ dLdG, double cst, const double2 *wall, double2 *hall) {
    using C = double2;
    constexpr int NB = 3 * NA;
    const int s1 = (ch == 4) ? -1 : 1;
    const int s2 = (ch == 2) ? 1 : -1;
    const int N = t.N, nk = t.n_keys;
    const int domains = a.tri & *t.domains;
    extern __shared__ __align__(16) unsigned char smem[];
    C *sW = reinterpret_cast<C *>(smem);                        // [NB][nk][9]
    C *sZ = sW + NB * nk * 9;                                   // [NB * NB][kAdjLd]
    unsigned long long *sQ = reinterpret_cast<unsigned long long *>(sZ + NB * NB * kAdjLd);   // [kAdjThreads * NB]
    __shared__ unsigned long long s_scan[4];
    __shared__ int s_q2[kAdjThreads], s_j1[kAdjThreads];

    const int ml = blockIdx.x / N, q1 = blockIdx.x - ml * N;
    const int ms = mode0 + ml;
    const int m0 = a.modes[ms];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    const C *W = wall + (size_t)blockIdx.x * (NB * nk * 9);
    C *H = hall + (size_t)blockIdx.x * (NB * nk * 9);              // may be W's own place
    const double gl = dLdG[(size_t)ch * a.n_modes + ms] * cst;
    const unsigned vm1 = t.vmask[q1];
    for (int k = threadIdx.x; k < NB * nk * 9; k += kAdjThreads) {
        const int j = k / (nk * 9), rem = k - j * (nk * 9);
        sW[k] = paired_value(t.perm4, rem / 9, W + j * (nk * 9) + rem % 9, 9);
    }
    __syncthreads();                                             // the whole of W is read
    for (int k = threadIdx.x; k < NB * nk * 9; k += kAdjThreads) H[k] = czero<C>();
    if ((q0 == 0 && j0 < 3) || gl == 0.0 || !vm1) return;
    const int4 c0 = t.qc[q0], c1 = t.qc[q1];
    const int b0 = c0.x + s1 * c1.x, b1 = c0.y + s1 * c1.y, b2 = c0.z + s1 * c1.z;
    const double w0 = t.om[m0];
    const float w0f = t.om32[m0];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;

    for (int qb = 0; qb < N; qb += kAdjThreads) {
        // window: one q'' per thread against every j'; entries of a j' are consecutive in the queue.
        // The scan runs over the NB <= 6 counts (0 or 1 a thread, at most 128 a round) packed in 10 bits.
        const int q2 = qb + threadIdx.x;
        unsigned long long ent[NB], cnt = 0;
#pragma unroll
        for (int j1 = 0; j1 < NB; ++j1) ent[j1] = 0;
        if (q2 < N) {
            const int4 c2 = t.qc[q2];
            const int q3 = q_index(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z, t.mesh[0], t.mesh[1], t.mesh[2]);
            const int tri = tri_code(domains, ch, q1, q2, q3);
            if (tri >= 0)
#pragma unroll
                for (int j1 = 0; j1 < NB; ++j1) {
                    if (!((vm1 >> j1) & 1u)) continue;
                    const int m1 = q1 * NB + j1;
                    unsigned mask[NB];
                    if (window_masks<NB, ADA>(t, a, domains, ch, s2, w0f + (float)s1 * t.om32[m1], m0, m1, w0, t.om[m1], q2, q3,
                                              mask) == 0)
                        continue;
                    unsigned long long e = ((unsigned long long)threadIdx.x << 48) | ((unsigned long long)j1 << 40) |
                                           ((unsigned long long)tri << 36);
#pragma unroll
                    for (int j3 = 0; j3 < NB; ++j3) e |= (unsigned long long)mask[j3] << (NB * j3);
                    ent[j1] = e;
                    cnt |= 1ull << (10 * j1);
                }
        }
        unsigned long long x = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_scan[wid] = x;
        __syncthreads();                                         // also orders sW, sQ
        unsigned long long before = x - cnt, all = 0;
        for (int w = 0; w < kAdjThreads / 32; ++w) {
            if (w < wid) before += s_scan[w];
            all += s_scan[w];
        }
        int total = 0;
#pragma unroll
        for (int j1 = 0; j1 < NB; ++j1) {
            if ((cnt >> (10 * j1)) & 1u) sQ[total + (int)((before >> (10 * j1)) & 1023u)] = ent[j1];
            total += (int)((all >> (10 * j1)) & 1023u);
        }
        __syncthreads();

        for (int first = 0; first < total; first += kAdjThreads) {
            const int n = min(kAdjThreads, total - first);
            if ((int)threadIdx.x < n) {
                const unsigned long long e = sQ[first + threadIdx.x];
                const int iq2 = qb + (int)(e >> 48), j1 = (int)((e >> 40) & 0xff), tri = (int)((e >> 36) & 3u);
                const int4 cc2 = t.qc[iq2];
                const int iq3 = q_index(b0 + s2 * cc2.x, b1 + s2 * cc2.y, b2 + s2 * cc2.z, t.mesh[0], t.mesh[1], t.mesh[2]);
                const int m1 = q1 * NB + j1;
                s_q2[threadIdx.x] = iq2;
                s_j1[threadIdx.x] = j1;
                const C *Prow = t.P4 + (size_t)iq2 * nk, *Wj = sW + j1 * nk * 9;
                C *Z = sZ + threadIdx.x;
                C X[NA][NA][9];
#pragma unroll
                for (int c = 0; c < NA; ++c)
#pragma unroll
                    for (int d = 0; d < NA; ++d)
                        paired_sum(t.perm4, t.grp_start[c * NA + d], t.pairs4[c * NA + d], t.grp_start[c * NA + d + 1], Prow, Wj,
                                   (double)s2, X[c][d]);
                const C *e2row = t.ev + (size_t)iq2 * NB * NB, *e3row = t.ev + (size_t)iq3 * NB * NB;
                const double w01 = (ch == 4 ? 1.0 / 6.0 : 0.5) * gl * t.invw[m0] * t.invw[m1];
                const double w1 = t.om[m1], n1 = t.occ[m1];
                bool started = false;
                unsigned rows = 0;                               // each lane goes through its own items
#pragma unroll
                for (int j3 = 0; j3 < NB; ++j3)
                    if ((unsigned)(e >> (NB * j3)) & ((1u << NB) - 1u)) rows |= 1u << j3;
                while (rows) {
                    const int j3 = __ffs(rows) - 1;
                    rows &= rows - 1;
                    unsigned m = (unsigned)(e >> (NB * j3)) & ((1u << NB) - 1u);
                    C Y[NB], yb[NB];
#pragma unroll
                    for (int k = 0; k < NB; ++k) Y[k] = yb[k] = czero<C>();
#pragma unroll
                    for (int d = 0; d < NA; ++d)
#pragma unroll
                        for (int dl = 0; dl < 3; ++dl) {
                            const C e3 = cconj(e3row[(3 * d + dl) * NB + j3]);
#pragma unroll
                            for (int c = 0; c < NA; ++c)
#pragma unroll
                                for (int g = 0; g < 3; ++g) Y[3 * c + g] = cfma(X[c][d][3 * g + dl], e3, Y[3 * c + g]);
                        }
                    const int m3 = iq3 * NB + j3;
                    while (m) {
                        const int j2 = __ffs(m) - 1;
                        m &= m - 1;
                        const int m2 = iq2 * NB + j2;
                        C V = czero<C>();
#pragma unroll
                        for (int k = 0; k < NB; ++k) V = cfma(cconj_if(e2row[k * NB + j2], s2 < 0), Y[k], V);
                        const double d = delta_exact(ch, w0, w1, t.om[m2], t.om[m3]);
                        double gs;
                        if constexpr (ADA) gs = gauss_adaptive(t, a, d, m2, m3);
                        else gs = exp(-(d * d) * a.inv_sigma2) * a.gnorm;
                        double w = w01 * occupation_factor<double>(ch, n1, t.occ[m2], t.occ[m3]) * gs * t.invw[m2] *
                                   t.invw[m3];
                        // the swapped process is added with the swapped legs; a self-swapped one counts half
                        if ((tri == 2 && j2 == j3) || (tri == 3 && j2 == j1)) w *= 0.5;
                        const C f = cmake(w * V.x, -w * V.y);                           // G conj(V)
#pragma unroll
                        for (int k = 0; k < NB; ++k) yb[k] = cfma(f, cconj_if(e2row[k * NB + j2], s2 < 0), yb[k]);
                    }
#pragma unroll
                    for (int dk = 0; dk < NB; ++dk) {
                        const C e3 = cconj(e3row[dk * NB + j3]);
#pragma unroll
                        for (int k = 0; k < NB; ++k) {
                            C *z = Z + (k * NB + dk) * kAdjLd;
                            *z = started ? cfma(yb[k], e3, *z) : cmul(yb[k], e3);
                        }
                    }
                    started = true;
                }
            }
            __syncthreads();
            // H_r[j'][γδ] += Σ P_r^s2 Z[c_r γ, d_r δ] over this batch, j' by j', in queue order; of a pair of
            // mirror keys the first collects Σ cos θ Z and the second Σ s2 sin θ Z
            for (int k = threadIdx.x; k < nk * 9; k += kAdjThreads) {
                const int p = k / 9, gd = k - 9 * p, g = gd / 3, dl = gd - 3 * g;
                const int e = t.perm4[p], kind = e >> 28, r = e & kKeyMask;
                const int rp = kind == 2 ? t.perm4[p - 1] & kKeyMask : r;        // the key whose phase it takes
                int grp = 0;
                while (t.grp_start[grp + 1] <= r) ++grp;
                const C *Z = sZ + ((3 * (grp / NA) + g) * NB + 3 * (grp % NA) + dl) * kAdjLd;
                for (int i = 0; i < n;) {
                    const int j1 = s_j1[i];
                    C h = H[(j1 * nk + r) * 9 + gd];
                    if (kind == 0) {
                        for (; i < n && s_j1[i] == j1; ++i)
                            h = cfma(cconj_if(t.P4[(size_t)s_q2[i] * nk + rp], s2 < 0), Z[i], h);
                    } else {
                        for (; i < n && s_j1[i] == j1; ++i) {
                            const C ph = t.P4[(size_t)s_q2[i] * nk + rp];
                            h = crfma(kind == 1 ? ph.x : s2 * ph.y, Z[i], h);
                        }
                    }
                    H[(j1 * nk + r) * 9 + gd] = h;
                }
            }
            __syncthreads();
        }
    }
    // pairs: H_dR = A + i B, H_-dR = A - i B
    for (int k = threadIdx.x; k < NB * nk * 9; k += kAdjThreads) {
        const int j = k / (nk * 9), rem = k - j * (nk * 9), p = rem / 9, gd = rem - 9 * p;
        if (t.perm4[p] >> 28 != 1) continue;
        C *x = H + (j * nk + (t.perm4[p] & kKeyMask)) * 9 + gd, *y = H + (j * nk + (t.perm4[p + 1] & kKeyMask)) * 9 + gd;
        const C A = *x, B = *y;
        *x = cmake(A.x - B.y, A.y + B.x);
        *y = cmake(A.x + B.y, A.y - B.x);
    }
}

constexpr int kFoldThreads = 256, kFoldAcc = 24;                 // 27 sums a cluster, 24 a thread

template <int NA>
__global__ void __launch_bounds__(kFoldThreads)
adj4_fold_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch, int mode0,
                 const double *__restrict__ dLdG, const double2 *__restrict__ hall, double *dphi_part) {
    using C = double2;
    constexpr int NB = 3 * NA;
    const int s1 = (ch == 4) ? -1 : 1;
    const int N = t.N, nk = t.n_keys, nc4 = t.nc4;
    extern __shared__ __align__(16) unsigned char smem[];
    C *sK = reinterpret_cast<C *>(smem);                        // [nk][NA][27]
    C *sPh = sK + nk * NA * 27;                                 // [nc4] phase / sqrt(m)
    C *sE1 = sPh + nc4;                                         // [NB][NB] e^s1_λ'(comp) per j'
    int *sSlot = reinterpret_cast<int *>(sE1 + NB * NB);         // [nc4] 27 (key NA + leg-1 atom) of a cluster
    const int ml = blockIdx.x, ms = mode0 + ml;
    const int m0 = a.modes[ms];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    const int out0 = blockIdx.y * (kFoldThreads * kFoldAcc);     // first of this block's 27 nc4 sums
    double *dphi = dphi_part + (size_t)ms * nc4 * 81;
    const int4 c0 = t.qc[q0];
    const bool active = !((q0 == 0 && j0 < 3) || dLdG[(size_t)ch * a.n_modes + ms] == 0.0);
    for (int rb = threadIdx.x; rb < nk * NA; rb += kFoldThreads)
        for (int i = t.kb_start[rb]; i < t.kb_start[rb + 1]; ++i) sSlot[t.kb_idx[i]] = 27 * rb;
    C acc[kFoldAcc];
#pragma unroll
    for (int i = 0; i < kFoldAcc; ++i) acc[i] = czero<C>();
    for (int q1 = 0; active && q1 < N; ++q1) {
        const int4 c1 = t.qc[q1];
        const C *H = hall + ((size_t)ml * N + q1) * (NB * nk * 9);
        __syncthreads();                                         // previous q' done
        for (int c = threadIdx.x; c < nc4; c += kFoldThreads) {
            const C ph = t.rt[mod_pos(s1 * phase_index(c1, t.c4_r13[c], t.L) - phase_index(c0, t.c4_r3[c], t.L), t.L)];
            sPh[c] = cmake(ph.x * t.c4_ism[c], ph.y * t.c4_ism[c]);
        }
        for (int k = threadIdx.x; k < NB * NB; k += kFoldThreads) {
            const int j1 = k / NB, comp = k - j1 * NB;
            sE1[k] = cconj_if(t.ev[((size_t)q1 * NB + comp) * NB + j1], s1 < 0);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < nk * 9; k += kFoldThreads) {
            const int r = k / 9, gd = k - 9 * r;
            C h[NB];
#pragma unroll
            for (int j1 = 0; j1 < NB; ++j1) h[j1] = H[j1 * nk * 9 + k];
#pragma unroll
            for (int bb = 0; bb < NB; ++bb) {
                C s = cmul(sE1[bb], h[0]);
#pragma unroll
                for (int j1 = 1; j1 < NB; ++j1) s = cfma(sE1[j1 * NB + bb], h[j1], s);
                sK[(r * NA + bb / 3) * 27 + (bb % 3) * 9 + gd] = s;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kFoldAcc; ++i) {
            const int o = out0 + i * kFoldThreads + threadIdx.x;
            if (o < nc4 * 27) {
                const int c = o / 27;
                acc[i] = cfma(sPh[c], sK[sSlot[c] + o - 27 * c], acc[i]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kFoldAcc; ++i) {
        const int o = out0 + i * kFoldThreads + threadIdx.x;
        if (o < nc4 * 27) {
            const int c = o / 27, k = o - 27 * c, a0 = t.c4_at[c].x;
#pragma unroll
            for (int al = 0; al < 3; ++al) {
                const C e0 = t.ev[((size_t)q0 * NB + 3 * a0 + al) * NB + j0];
                dphi[(size_t)c * 81 + 27 * al + k] = 2.0 * (e0.x * acc[i].x - e0.y * acc[i].y);
            }
        }
    }
}

// ------------------------------------------------------------------------------ three-phonon

// One block per mode.  The processes wait in the rate kernel's queue; a round of 128 evaluates one
// process per thread (V3 from the mode's cluster sums G) and leaves G conj(V) e^s_λ' and e*_λ'' in shared
// memory, from which the owner of each (key r, βγ) adds P_r(q')^s e^s_λ'(bβ) e*_λ''(cγ) G conj(V) to
//   H_r[βγ] = dL/dG_r[βγ]  (processes in queue order),
// and the mode's gradient slice is 2 Re(exp(-i q.R2) e_λ(aα) H_r(c)[βγ]) / sqrt(m).
// Bound: FP64 (966 complex multiply-adds a process for the diamond cell); adding to all 27 nc3 entries
// process by process took 12.8 ms for the 384 modes of a 4^3 mesh.
// GLOBAL: G and H of more keys than shared memory holds (adj3_scratch_per_mode) lie in a.gh3, a part for each mode.
template <int NA, bool ADA, bool GLOBAL>
__global__ void __launch_bounds__(kR3Threads)
adj3_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch,
            const double *__restrict__ dLdG, double cst, double *dphi_part) {
    constexpr int NB = 3 * NA, JB = jb3(NB), LD = kR3Threads + 1;
    using C = double2;
    const int N = t.N, nc3 = t.nc3, nk = t.n_keys3;
    extern __shared__ __align__(16) unsigned char smem[];
    C *sG = GLOBAL ? a.gh3 + (size_t)blockIdx.x * (nk * 18) : reinterpret_cast<C *>(smem);   // [nk][9]
    C *sH = sG + nk * 9;                                        // [nk][9]
    C *sE = GLOBAL ? reinterpret_cast<C *>(smem) : sH + nk * 9; // [2 NB][LD] G conj(V) e^s_λ' and e*_λ''
    unsigned *sList = reinterpret_cast<unsigned *>(sE + 2 * NB * LD);
    __shared__ C se0[NB];
    __shared__ int s_scan[32], s_q1[kR3Threads];
    const int ms = blockIdx.x;
    const Three p(t, ch, a.modes[ms], NB);
    double *dphi = dphi_part + (size_t)ms * nc3 * 27;
    const double gl = dLdG[(size_t)ch * a.n_modes + ms] * cst;
    if ((p.q0 == 0 && p.j0 < 3) || gl == 0.0) {
        for (int k = threadIdx.x; k < nc3 * 27; k += kR3Threads) dphi[k] = 0.0;
        return;
    }
    for (int k = threadIdx.x; k < NB; k += kR3Threads) se0[k] = t.ev[(p.q0 * NB + k) * NB + p.j0];
    __syncthreads();
    three_G<false>(t, p, se0, sG);
    for (int k = threadIdx.x; k < nk * 9; k += kR3Threads) sH[k] = czero<C>();
    auto round = [&](int qlo, int first, int n) {
        if ((int)threadIdx.x < n) {
            const ThreeProcess z = three_evaluate<NA, ADA>(t, a, p, qlo, sList[first + threadIdx.x], sG);
            const C f = cmake(gl * z.w * z.V.x, -gl * z.w * z.V.y);                     // G conj(V)
            s_q1[threadIdx.x] = z.q1;
#pragma unroll 1
            for (int k = 0; k < NB; ++k) {
                sE[k * LD + threadIdx.x] = cmul(f, cconj_if(t.ev[((size_t)z.q1 * NB + k) * NB + z.j1], p.s < 0));
                sE[(NB + k) * LD + threadIdx.x] = cconj(t.ev[((size_t)z.q2 * NB + k) * NB + z.j2]);
            }
        }
        __syncthreads();
        for (int k = threadIdx.x; k < nk * 9; k += kR3Threads) {
            const int r = k / 9, bg = k - 9 * r, be = bg / 3, g = bg - 3 * be;
            int grp = 0;
            while (t.grp3_start[grp + 1] <= r) ++grp;
            const C *x = sE + (3 * (grp / NA) + be) * LD, *y = sE + (NB + 3 * (grp % NA) + g) * LD;
            C h = sH[k];
            for (int i = 0; i < n; ++i)
                h = cfma(cmul(cconj_if(t.P3[(size_t)s_q1[i] * nk + r], p.s < 0), x[i]), y[i], h);
            sH[k] = h;
        }
        __syncthreads();
    };
    for (int qlo = 0; qlo < N; qlo += kQueueSpan3) {                // the queue is empty between spans
        const int qhi = min(N, qlo + kQueueSpan3);
        int queued = 0;
        for (int qb = qlo; qb < qhi; qb += kR3Threads)
            for (int jb = 0; jb < NB; jb += JB) {
                queued = three_append<NB, ADA, JB>(t, a, p, qlo, qb, qhi, jb, queued, sList, s_scan);
                for (; queued >= kR3Threads; queued -= kR3Threads) round(qlo, queued - kR3Threads, kR3Threads);
            }
        if (queued) round(qlo, 0, queued);
    }
    for (int r = 0; r < nk; ++r) {
        const int i0 = t.k3_start[r], n = (t.k3_start[r + 1] - i0) * 27;
        for (int k = threadIdx.x; k < n; k += kR3Threads) {
            const int c = t.k3_idx[i0 + k / 27], abg = k % 27, al = abg / 9, bg = abg - 9 * al;
            const C ph = cconj(t.rt[phase_index(p.c0, t.c3_r2[c], t.L)]);
            const C z = cmul(cmul(ph, se0[3 * t.c3_at[c].x + al]), sH[r * 9 + bg]);
            dphi[(size_t)c * 27 + abg] = 2.0 * t.c3_ism[c] * z.x;
        }
    }
}

// Shared memory of the 3ph adjoint beside G and H: the processes of a round and their queue.
static size_t adj3_lists_smem(int na) {
    const int nb = 3 * na;
    return sizeof(double2) * (size_t)2 * nb * (kR3Threads + 1) + sizeof(unsigned) * (size_t)kR3Threads * (jb3(nb) * nb + 1);
}

// 288 bytes of G and H a key: up to 650 keys (two atoms; four: 565) in shared memory, beyond that in device memory
// (a block's G and H stay in L2).  Clusters with a key each, one q, cluster by cluster and now: two atoms, 5^3, 500
// clusters 44 and 4.1 ms, 700 (in device memory) 62 and 6.0 ms; four atoms, 3^3, 1500 clusters 566 and 74 ms.
size_t adj3_scratch_per_mode(const Tables &t) {
    const size_t gh = sizeof(double2) * (size_t)t.n_keys3 * 18;
    return t.n_atoms <= 4 && gh + adj3_lists_smem(t.n_atoms) > 226 * 1024 ? gh : 0;
}

// ------------------------------------------------------------------------------ slices -> gradient

// out (+)= Σ_slices part in slice order; with swap set (Φ4 entries, 81 a cluster), and where Φ4 still has that
// symmetry, each slice also adds the entry of the cluster with two legs exchanged (twelve: legs 1 and 2, else 2 and 3).
__global__ void sum_slices_kernel(int n_slices, int n, const double *part, double *out, int accumulate,
                                  int kahan32, const int *swap, int twelve, const int *domains) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double s = accumulate ? out[k] : 0.0;
    if (kahan32) {                                       // FP32 (sum, compensation) pairs
        const float2 *p = reinterpret_cast<const float2 *>(part);
        for (int i = 0; i < n_slices; ++i) {
            const float2 v = p[(size_t)i * n + k];
            s += (double)v.x - (double)v.y;
        }
    } else {
        for (int i = 0; i < n_slices; ++i) s += part[(size_t)i * n + k];
        if (swap && (*domains & (twelve ? 2 : 1))) {
            const int c = k / 81, e = k - 81 * c;
            const int al = e / 27, x = (e / 9) % 3, y = (e / 3) % 3, z = e % 3;
            const int o = 81 * swap[c] + (twelve ? ((al * 3 + y) * 3 + x) * 3 + z : ((al * 3 + x) * 3 + z) * 3 + y);
            for (int i = 0; i < n_slices; ++i) s += part[(size_t)i * n + o];
        }
    }
    out[k] = s;
}

// Shared memory of the tiled FP64 adjoint's unit kernel.
template <int NA>
static size_t adj4_tile_smem(const Tables &t) {
    constexpr int NB = 3 * NA;
    return sizeof(double2) * ((size_t)NB * t.n_keys * 9 + (size_t)NB * NB * kAdjLd) +
           sizeof(unsigned long long) * (size_t)kAdjThreads * NB;
}

template <int NA>
static size_t adj4_fold_smem(const Tables &t) {
    return sizeof(double2) * ((size_t)t.n_keys * NA * 27 + t.nc4 + 9 * NA * NA) + sizeof(int) * (size_t)t.nc4;
}

// The tiled path serves FP64 cells of up to two atoms whose tables fit in shared memory, those of its W included.
template <int NA>
static bool adj4_fits(const Tables &t) {
    constexpr size_t most = 220 * 1024;
    return adj4_tile_smem<NA>(t) <= most && adj4_fold_smem<NA>(t) <= most && w4_smem_bytes<double, NA>(t) <= kW4MostSmem;
}

bool adj4_tiled(const Tables &t) {
    return t.n_atoms == 1 ? adj4_fits<1>(t) : t.n_atoms == 2 && adj4_fits<2>(t);
}

template <int NA, bool ADA>
static cudaError_t launch_adj4_tile(const Tables &t, const RateArgs &a, int ch, const double *dLdG, double cst,
                                    double *part, cudaStream_t s) {
    const size_t per_mode = tile_w_bytes_per_mode<double, NA>(t);
    const int chunk = (int)std::min<size_t>(a.wbuf_bytes / per_mode, 0x7fffffffu / (unsigned)t.N);
    if (chunk < 1) return cudaErrorInvalidValue;
    const size_t smem = adj4_tile_smem<NA>(t), fsmem = adj4_fold_smem<NA>(t);
    // with a place of its own for H, W stays and +- takes the one of ++ (w_reuse)
    const bool both = a.hbuf && chunk >= a.n_modes;
    double2 *w = reinterpret_cast<double2 *>(a.wbuf), *h = both ? reinterpret_cast<double2 *>(a.hbuf) : w;
    cudaError_t e = cudaFuncSetAttribute(adj4_tile_kernel<NA, ADA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(adj4_fold_kernel<NA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsmem);
    if (e != cudaSuccess) return e;
    const int n_out = (27 * t.nc4 + kFoldThreads * kFoldAcc - 1) / (kFoldThreads * kFoldAcc);
    for (int m = 0; m < a.n_modes; m += chunk) {
        const int nm = std::min(chunk, a.n_modes - m);
        if (!(both && a.w_reuse)) e = launch_w4<double, NA>(t, a, ch, m, nm, s);
        if (e != cudaSuccess) return e;
        adj4_tile_kernel<NA, ADA><<<(unsigned)((long long)nm * t.N), kAdjThreads, smem, s>>>(t, a, ch, m, dLdG, cst, w, h);
        adj4_fold_kernel<NA><<<dim3(nm, n_out), kFoldThreads, fsmem, s>>>(t, a, ch, m, dLdG, h, part);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int NA>
static cudaError_t launch_adj_na(const Tables &t, const RateArgs &a, int ch, const double *dLdG, double cst,
                                 double *part, int fp64, cudaStream_t s) {
    if (a.n_modes == 0) return cudaSuccess;
    if (ch < 2) {
        const bool global = adj3_scratch_per_mode(t) != 0;
        if (global && !a.gh3) return cudaErrorInvalidValue;
        const size_t gh = sizeof(double2) * (size_t)t.n_keys3 * 18, smem = adj3_lists_smem(NA) + (global ? 0 : gh);
        auto kern = global ? (a.adaptive ? adj3_kernel<NA, true, true> : adj3_kernel<NA, false, true>)
                           : (a.adaptive ? adj3_kernel<NA, true, false> : adj3_kernel<NA, false, false>);
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<a.n_modes, kR3Threads, smem, s>>>(t, a, ch, dLdG, cst, part);
        return cudaGetLastError();
    }
    if constexpr (NA <= 2)
        if (fp64 && a.wbuf)
            return a.adaptive ? launch_adj4_tile<NA, true>(t, a, ch, dLdG, cst, part, s)
                              : launch_adj4_tile<NA, false>(t, a, ch, dLdG, cst, part, s);
    auto run = [&](auto zero) -> cudaError_t {
        using R = decltype(zero);
        using C = Cplx<R>;
        constexpr int NB = 3 * NA;
        const size_t smem = sizeof(C) * ((size_t)t.n_keys * 18 + (size_t)t.nc4 * 10 + NA * NA * 9 + NB) +
                            sizeof(Item4<R, NA>) * kAdjThreads + 16;
        cudaError_t e = cudaFuncSetAttribute(adj4_kernel<R, NA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        adj4_kernel<R, NA><<<a.n_modes, kAdjThreads, smem, s>>>(t, a, ch, dLdG, cst, part);
        return cudaGetLastError();
    };
    return fp64 ? run(0.0) : run(0.0f);
}

cudaError_t launch_adjoint(const Tables &t, const RateArgs &a, int ch, const double *dLdG, double cst,
                           double *part, int fp64, cudaStream_t s) {
    switch (t.n_atoms) {
    case 1: return launch_adj_na<1>(t, a, ch, dLdG, cst, part, fp64, s);
    case 2: return launch_adj_na<2>(t, a, ch, dLdG, cst, part, fp64, s);
    case 3: return launch_adj_na<3>(t, a, ch, dLdG, cst, part, fp64, s);
    case 4: return launch_adj_na<4>(t, a, ch, dLdG, cst, part, fp64, s);
    default: return cudaErrorInvalidValue;       // cells of more than 4 atoms: not instantiated
    }
}

cudaError_t launch_sum_slices(int n_slices, int n, const double *part, double *out, int accumulate,
                              int kahan32, const int *swap, int twelve, const int *domains, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    sum_slices_kernel<<<(n + 63) / 64, 64, 0, s>>>(n_slices, n, part, out, accumulate, kahan32, swap, twelve, domains);
    return cudaGetLastError();
}

}  // namespace fc4
