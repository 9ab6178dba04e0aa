// k_rates4_tile.cuh - four-phonon path for small cells (<= 2 atoms), in two kernels.
//
// w4_kernel writes W_r[γδ](λ, q', j') for every partner branch j' of a unit (λ, q') to a global
// buffer (HBM is otherwise idle here; one pass over the clusters per unit).  rates4_tile_kernel
// then owns the unit: it copies that W to shared memory, sweeps q'' in rounds of 128 threads x
// kQPT q'' (over the unit's triangle where the partner-swap symmetry holds), tests the window
// against every j' at once (branch-free FP32 prefilter, rare ambiguous candidates decided by the
// exact FP64 Δ), compacts the (q'', j', masks) entries with a block scan, and evaluates them:
//   X[c,d][γδ] = Σ_{r in (c,d)} P_r^s2 W_r[γδ] once per entry, Y = X e*''' per j''' (36 MACs).
// FP64 holds X too (2 blocks of 255 registers per SM; with one atom, whose X is a quarter, 3 blocks: all modes of
// 3^3, ++, 149 -> 110 us): its pipe issues a warp operation every ~19 clocks and SM, so what counts is the
// 198 + 36 items complex multiply-adds of an entry (306 + 36 items without the pairing of mirror keys), against
// 408 an item key by key.
// The same window decision, weights and accumulation as the general kernel (k_rates4.cuh).
#pragma once
#include "k_rates4.cuh"

namespace fc4 {

constexpr int kTileQ = 128;
// Partner points q'' per thread and compaction round, and blocks per SM.  Fixed σ: 4 for the
// sparse ++ and -- channels (more window work per round), 2 for +- (fewer registers held across
// its dense entry work), 4 blocks of 128 threads per SM (128 registers).  Adaptive σ carries the
// pair widths and the per-process width through the same loops: at 128 registers it spilled
// (~500 bytes), so it runs 3 blocks per SM (168 registers) with 2 and 1 q'' per round; measured on
// the 16^3 precision workload this took a 5-q batch from 792 to 614 ms, while the fixed-σ kernels
// lose 1-3 % with either change (the adaptive ++ and --, which now hold no widths, still take 90 ms so and 97
// at 4 blocks: two q of 16^3).
constexpr int kQPTSparse = 4, kQPTDense = 2;
constexpr int kQPTSparseAd = 2, kQPTDenseAd = 1;
template <bool ADA> constexpr int qpt_of(bool dense) {
    return ADA ? (dense ? kQPTDenseAd : kQPTSparseAd) : (dense ? kQPTDense : kQPTSparse);
}
// q'' per chunk of the +- triangle list (the q'' <= q''' of a unit, built in shared memory)
constexpr int kTriChunk = 1024;


// W[j'][r][γδ] of units (λ, q') for every partner branch j', written to global memory (layout
// [unit][j'][r][γδ]).  One block per (λ, group of kW4Group q'): Φ contracted with e_λ and the mass
// factor, Φ~_c[β][γδ] = Σ_α Φ_c[αβγδ] e_λ(aα) / sqrt(m), is built once in shared memory.  Per q' the
// cluster phases are folded first, per key r and leg-1 atom b,
//   Ψ_rb[β][γδ] = Σ_{c in r, b(c) = b} exp(i(s1 q'.(R1 - R3) - q.R3)) Φ~_c[β][γδ]   (fixed order),
// and then W_r[γδ] = Σ_b Σ_β e^s1_λ'(bβ) Ψ_rb[β][γδ] for every j' (coalesced writes): the phase
// work is shared by all partner branches.  FP64: the work is spread evenly over the threads, which the FP64
// pipe needs (4.7 ms for both signs of 4 q points of 8^3, against 5.7 ms for the column kernel below).
constexpr int kW4Group = 8;

constexpr int kW4Threads = 256;

template <typename R, int NA>
__global__ void __launch_bounds__(kW4Threads)
w4_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch, int mode0,
          Cplx<R> *wout) {
    using C = Cplx<R>;
    constexpr int NB = 3 * NA;
    const int s1 = (ch == 4) ? -1 : 1;
    const int N = t.N, nk = t.n_keys, nc4 = t.nc4;
    const int ngrp = (N + kW4Group - 1) / kW4Group;
    extern __shared__ __align__(16) unsigned char smem[];
    C *sPt = reinterpret_cast<C *>(smem);                       // [nc4][3][9]
    C *sPh = sPt + nc4 * 27;                                    // [nc4]
    C *sE1 = sPh + nc4;                                         // [NB][NB]  e^s1_λ'(comp) per j'
    C *se0 = sE1 + NB * NB;                                     // [NB]
    C *sPsi = se0 + NB;                                         // [nk][NA][27]
    const int ml = blockIdx.x / ngrp, qg = blockIdx.x - ml * ngrp;
    const int m0 = a.modes[mode0 + ml];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    const C *ev = Sel<R>::ev(t);
    const C *rt = Sel<R>::rt(t);
    const R *phi4 = Sel<R>::phi4(t);
    const R *ism4 = Sel<R>::ism4(t);
    const int4 c0 = t.qc[q0];
    for (int k = threadIdx.x; k < NB; k += blockDim.x) se0[k] = ev[(q0 * NB + k) * NB + j0];
    __syncthreads();
    for (int k = threadIdx.x; k < nc4 * 27; k += blockDim.x) {
        const int c = k / 27, rem = k - c * 27;
        const int be = rem / 9, gd = rem - be * 9;
        const int a0 = t.c4_at[c].x;
        const R *ph4 = phi4 + 81 * c + be * 9 + gd;
        C v = czero<C>();
#pragma unroll
        for (int al = 0; al < 3; ++al) v = crfma(ph4[27 * al], se0[3 * a0 + al], v);
        sPt[k] = cmake(v.x * ism4[c], v.y * ism4[c]);
    }
    const int q1_end = min(N, (qg + 1) * kW4Group);
    for (int q1 = qg * kW4Group; q1 < q1_end; ++q1) {
        const int4 c1 = t.qc[q1];
        __syncthreads();                                         // sPt ready / previous q' done
        for (int c = threadIdx.x; c < nc4; c += blockDim.x)
            sPh[c] = rt[mod_pos(s1 * phase_index(c1, t.c4_r13[c], t.L) - phase_index(c0, t.c4_r3[c], t.L), t.L)];
        for (int k = threadIdx.x; k < NB * NB; k += blockDim.x) {
            const int j1 = k / NB, comp = k - j1 * NB;
            sE1[k] = cconj_if(ev[(q1 * NB + comp) * NB + j1], s1 < 0);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < nk * NA * 27; k += blockDim.x) {
            const int rb = k / 27, bgd = k - rb * 27;            // rb = r NA + b
            C acc = czero<C>();
            for (int i = t.kb_start[rb]; i < t.kb_start[rb + 1]; ++i) {
                const int c = t.kb_idx[i];
                acc = cfma(sPh[c], sPt[c * 27 + bgd], acc);
            }
            sPsi[k] = acc;
        }
        __syncthreads();
        C *wo = wout + ((size_t)ml * N + q1) * NB * nk * 9;
        for (int k = threadIdx.x; k < NB * nk * 9; k += blockDim.x) {
            const int j1 = k / (nk * 9), rem = k - j1 * (nk * 9);
            const int r = rem / 9, gd = rem - r * 9;
            const C *e1 = sE1 + j1 * NB;
            const C *ps = sPsi + r * NA * 27 + gd;
            C acc = czero<C>();
#pragma unroll
            for (int b = 0; b < NA; ++b)
#pragma unroll
                for (int be = 0; be < 3; ++be) acc = cfma(e1[3 * b + be], ps[b * 27 + be * 9], acc);
            wo[k] = acc;
        }
    }
}

// The same in FP32, for a group of q' per block: a thread owns a column (r, γδ) for kW4Pair q' at a time.
// It folds the cluster phases into its six
//   Ψ_rb[β][γδ] = Σ_{c in r, b(c) = b} exp(i(s1 q'.(R1 - R3) - q.R3)) Φ~_c[β][γδ]   (fixed order)
// in registers and writes W_r[γδ] = Σ_b Σ_β e^s1_λ'(bβ) Ψ_rb[β][γδ] for every j' (the same sums in the
// same order).
//
// Bound: FP32 issue and shared-memory loads; 17000 complex multiply-adds a unit (the 14.7 KB a unit
// written take an eighth of the time).  Ψ in registers needs no barrier between the two sums, and a
// column reads its six Ψ once for all j' and its Φ~ once for two q'; keys are taken from the
// longest cluster list down, so that the two keys with R2 = R3 (49 of 226 clusters each, the others 4)
// share a warp, which moves over the warps from block to block.  Both signs of all modes of 8^3:
// 29.3 ms, against 57 ms with Ψ in shared memory.
constexpr int kW4Pair = 2;

template <int NA>
struct W4Smem {
    using C = float2;
    static constexpr int NB = 3 * NA;
    C *Pt, *Ph, *E1, *e0;
    int *i3, *kb, *idx;
    __host__ __device__ static size_t bytes(const Tables &t) {
        return sizeof(C) * ((size_t)t.nc4 * 27 + (size_t)t.nc4 * kW4Pair + NB * NB * kW4Pair + NB) +
               sizeof(int) * ((size_t)2 * t.nc4 + (size_t)t.n_keys * NA + 1);
    }
    __device__ __forceinline__ W4Smem(unsigned char *smem, const Tables &t) {
        Ph = reinterpret_cast<C *>(smem);                       // [nc4][kW4Pair] phases
        E1 = Ph + t.nc4 * kW4Pair;                              // [kW4Pair][NB][NB] e^s1_λ'(comp) per j'
        Pt = E1 + NB * NB * kW4Pair;                            // [nc4][3][9]
        e0 = Pt + t.nc4 * 27;                                   // [NB]
        i3 = reinterpret_cast<int *>(e0 + NB);                  // [nc4] phase index of q.R3
        idx = i3 + t.nc4;                                       // [nc4] clusters by (key, leg-1 atom)
        kb = idx + t.nc4;                                       // [n_keys NA + 1] their ranges
    }
};

template <int NA>
__global__ void __launch_bounds__(384, 2)
w4_column_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch, int mode0, int group,
                 float2 *wout) {
    using C = float2;
    using R = float;
    constexpr int NB = 3 * NA;
    const int s1 = (ch == 4) ? -1 : 1;
    const int N = t.N, nk = t.n_keys, nc4 = t.nc4;
    const int ngrp = (N + group - 1) / group;
    extern __shared__ __align__(16) unsigned char smem[];
    const W4Smem<NA> sm(smem, t);
    const int ml = blockIdx.x / ngrp, qg = blockIdx.x - ml * ngrp;
    const int m0 = a.modes[mode0 + ml];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    const C *ev = Sel<R>::ev(t);
    const C *rt = Sel<R>::rt(t);
    const R *phi4 = Sel<R>::phi4(t);
    const R *ism4 = Sel<R>::ism4(t);
    const int4 c0 = t.qc[q0];
    for (int k = threadIdx.x; k < NB; k += blockDim.x) sm.e0[k] = ev[(q0 * NB + k) * NB + j0];
    for (int c = threadIdx.x; c < nc4; c += blockDim.x) {
        sm.i3[c] = phase_index(c0, t.c4_r3[c], t.L);
        sm.idx[c] = t.kb_idx[c];
    }
    for (int k = threadIdx.x; k <= nk * NA; k += blockDim.x) sm.kb[k] = t.kb_start[k];
    __syncthreads();
    for (int k = threadIdx.x; k < nc4 * 27; k += blockDim.x) {
        const int c = k / 27, rem = k - c * 27;
        const int a0 = t.c4_at[c].x;
        const R *ph4 = phi4 + 81 * c + rem;
        C v = czero<C>();
#pragma unroll
        for (int al = 0; al < 3; ++al) v = crfma(ph4[27 * al], sm.e0[3 * a0 + al], v);
        sm.Pt[k] = cmake(v.x * ism4[c], v.y * ism4[c]);
    }
    // the warp with the long keys sits on another scheduler in every block
    const int nw = blockDim.x >> 5;
    const int col0 = ((int)threadIdx.x + 32 * (int)(blockIdx.x % nw)) % (int)blockDim.x;
    const int q1_end = min(N, (qg + 1) * group);
    for (int q1 = qg * group; q1 < q1_end; q1 += kW4Pair) {
        const int nq = min(kW4Pair, q1_end - q1);
        __syncthreads();                                         // Pt ready / previous q' done
        for (int k = threadIdx.x; k < nc4 * kW4Pair; k += blockDim.x) {
            const int c = k / kW4Pair, qq = min(k - c * kW4Pair, nq - 1);
            const int4 c1 = t.qc[q1 + qq], r = t.c4_r13[c];
            sm.Ph[k] = rt[mod_pos(s1 * (c1.x * r.x + c1.y * r.y + c1.z * r.z) - sm.i3[c], t.L)];
        }
        for (int k = threadIdx.x; k < NB * NB * nq; k += blockDim.x) {
            const int qq = k / (NB * NB), rem = k - qq * NB * NB;
            const int j1 = rem / NB, comp = rem - j1 * NB;
            sm.E1[k] = cconj_if(ev[((q1 + qq) * NB + comp) * NB + j1], s1 < 0);
        }
        __syncthreads();
        for (int k = col0; k < nk * 9; k += blockDim.x) {
            const int r = t.key_order[k / 9], gd = k % 9;
            C psi[kW4Pair][NB];
#pragma unroll
            for (int qq = 0; qq < kW4Pair; ++qq)
#pragma unroll
                for (int bb = 0; bb < NB; ++bb) psi[qq][bb] = czero<C>();
#pragma unroll
            for (int b = 0; b < NA; ++b)
                for (int i = sm.kb[r * NA + b]; i < sm.kb[r * NA + b + 1]; ++i) {
                    const int c = sm.idx[i];
                    const C *pt = sm.Pt + c * 27 + gd;
                    C ph[kW4Pair];
#pragma unroll
                    for (int qq = 0; qq < kW4Pair; ++qq) ph[qq] = sm.Ph[c * kW4Pair + qq];
#pragma unroll
                    for (int be = 0; be < 3; ++be) {
                        const C x = pt[be * 9];
#pragma unroll
                        for (int qq = 0; qq < kW4Pair; ++qq) psi[qq][3 * b + be] = cfma(ph[qq], x, psi[qq][3 * b + be]);
                    }
                }
#pragma unroll
            for (int qq = 0; qq < kW4Pair; ++qq) {
                if (qq >= nq) break;
                C *wo = wout + (((size_t)ml * N + q1 + qq) * NB * nk + r) * 9 + gd;
                const C *e1 = sm.E1 + qq * NB * NB;
#pragma unroll
                for (int j1 = 0; j1 < NB; ++j1) {
                    C acc = czero<C>();
#pragma unroll
                    for (int bb = 0; bb < NB; ++bb) acc = cfma(e1[j1 * NB + bb], psi[qq][bb], acc);
                    wo[(size_t)j1 * nk * 9] = acc;
                }
            }
        }
    }
}

// BTE = true also accumulates the off-diagonal term of the iterative Boltzmann equation,
//   Δ_λ = Σ_p γ_p Σ_k s_k (ω_k / ω_λ) F_k  (partner signs: ++ (-, -, +), +- (-, +, +), -- (+, +, +)),
// into a.part_d; the partner combination is symmetric under the swap the triangular domain uses.
template <typename R, int NA, bool ADA, int kQPT, bool BTE = false, bool NOCOMP = false>
__global__ void __launch_bounds__(kTileQ, sizeof(R) == 8 ? (NA == 1 ? 3 : 2) : ADA ? 3 : 4)
rates4_tile_kernel(const __grid_constant__ Tables t, const __grid_constant__ RateArgs a, int ch,
                   int mode0, const Cplx<R> *__restrict__ wall) {
    using C = Cplx<R>;
    constexpr int NB = 3 * NA;
    constexpr bool WARP = sizeof(R) == 8 && !NOCOMP;
    constexpr bool SPARSE = kQPT == qpt_of<ADA>(false) && !NOCOMP;
    const int s1 = (ch == 4) ? -1 : 1;
    const int s2 = (ch == 2) ? 1 : -1;
    const int N = t.N, nk = t.n_keys;

    extern __shared__ __align__(16) unsigned char smem[];
    C *sW = reinterpret_cast<C *>(smem);                        // [NB][nk][9]
    unsigned long long *sQ = reinterpret_cast<unsigned long long *>(sW + NB * nk * 9);   // [kTileQ * NB * kQPT]
    // SPARSE: candidates [kTileQ * NB * kQPT] in the upper half of sQ (entry o is written after candidate
    // o + 127 has been read at the latest, so the two lists never meet)
    unsigned *sC = reinterpret_cast<unsigned *>(sQ) + kTileQ * NB * kQPT;
    float *s_g = reinterpret_cast<float *>(sQ + kTileQ * NB * kQPT);   // adaptive +-: [NB * NB][kTileQ] widths
    __shared__ int s_scan[32];
    __shared__ double s_red[(BTE ? 5 : 2) * 32];
    __shared__ long long s_redn[5 * 32];
    __shared__ unsigned short s_tri[kTriChunk];                 // +- triangle: q'' - chunk start
    // per warp, of one pass: its items (entry lane, j'''), their processes (item lane, j'') and the
    // processes' weight, weight |V|^2 (and BTE terms)
    constexpr int NV = BTE ? 5 : 2;
    __shared__ unsigned char s_item[WARP ? kTileQ * NB : 1], s_proc[WARP ? kTileQ * NB : 1];
    __shared__ R s_val[WARP ? kTileQ * NB * NV : 1];

    const int unit = blockIdx.x;                                // (mode - mode0) * N + q'
    const int ml = unit / N, q1 = unit - ml * N;
    const int ms = mode0 + ml;
    const int m0 = a.modes[ms];
    const int q0 = m0 / NB, j0 = m0 - q0 * NB;
    const C *ev = Sel<R>::ev(t);
    const C *P4 = Sel<R>::P4(t);
    const R *occ = Sel<R>::occ(t);
    const R *invw = Sel<R>::invw(t);

    Acc<R> acc_g, acc_wp;
    Acc<R> acc_d[BTE ? 3 : 1];
    long long acc_n = 0, acc_items = 0, acc_ent = 0, acc_ev = 0, acc_cev = 0;
    const unsigned vm1 = t.vmask[q1];

    if (!(q0 == 0 && j0 < 3) && vm1) {
        const int4 c0 = t.qc[q0], c1 = t.qc[q1];
        const int b0 = c0.x + s1 * c1.x, b1 = c0.y + s1 * c1.y, b2 = c0.z + s1 * c1.z;
        const double w0 = t.om[m0];
        const float w0f = t.om32[m0];
        // W of (λ, q') for every j'.  FP64: when the first entry turns up.  Many units of the sparse channels have
        // none, and with two blocks per SM nothing hides the copy (all modes of 3^3, FP64, ++: 409 -> 249 us, --:
        // 328 -> 161; two q of 6^3, +-: 1.69 ms either way).
        const C *src = wall + (size_t)unit * (NB * nk * 9);
        if constexpr (!WARP)
            for (int k = threadIdx.x; k < NB * nk * 9; k += kTileQ) sW[k] = src[k];
        bool have_w = !WARP;
        float base32[NB];
#pragma unroll
        for (int j = 0; j < NB; ++j) base32[j] = w0f + (float)s1 * t.om32[q1 * NB + j];

        // The triangular domain is walked without idle lanes: ++ and -- start at q'' = q'; +- takes
        // its q'' <= q''' from a list built per chunk of kTriChunk q'' (ascending order).
        const bool pm_list = (ch == 3) && (a.tri & 1);
        const int qstart = (ch != 3 && (a.tri & 2)) ? q1 : 0;
        for (int cb = qstart; cb < N; cb += pm_list ? kTriChunk : N) {
          int cnt = N - cb;
          if (pm_list) {
            constexpr int kPer = kTriChunk / kTileQ;
            const int ce = min(N, cb + kTriChunk), lo = cb + threadIdx.x * kPer;
            unsigned fl = 0;
            int nf = 0;
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int q2 = lo + i;
                if (q2 < ce) {
                    const int4 c2 = t.qc[q2];
                    const int q3 = q_index_near(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z,
                                                t.mesh[0], t.mesh[1], t.mesh[2]);
                    if (q2 <= q3) { fl |= 1u << i; ++nf; }
                }
            }
            int off = block_exclusive_scan(nf, s_scan, &cnt);
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                if ((fl >> i) & 1u) s_tri[off++] = (unsigned short)(threadIdx.x * kPer + i);
            __syncthreads();
          }
          for (int qb = 0; qb < cnt; qb += kTileQ * kQPT) {
            int total, n_ent = 0, off = 0;
            if constexpr (SPARSE) {
                const float wide = a.ad_rhi * a.ad_c32;          // adaptive: upper prefilter bound per unit of |ΔP|
                // ++, --: few (q'', j') have a pair near the window.  Pass 1 tests every q'' of the round with
                // cheap bounds and lists the (q'', j') left, in order; pass 2 takes that list one pair per
                // thread, so the mask work runs on full warps, and lists the entries (all modes of 8^3, ++ and
                // --: 126.6 -> 121.9 ms on top of the packed mode scalars, 112 with the loops as below; with the candidates in shared memory
                // of their own, which the L1 then lacks, it gained nothing).
                // Adaptive σ: no width exceeds the one of |P''| + |P'''|, and the pairs within that have theirs
                // formed in pass 2, one by one.  Two q of 16^3, both channels: 106.4 ms with the 36 widths of
                // every q'' kept in shared memory, 147 with one bound a q'', 90.0 with one a pair.
                unsigned cand[kQPT];
                int n_cand = 0;
#pragma unroll
                for (int k = 0; k < kQPT; ++k) {
                    cand[k] = 0;
                    const int q2 = cb + qb + k * kTileQ + (int)threadIdx.x;
                    if (q2 >= N) continue;
                    const int4 c2 = t.qc[q2];
                    const int q3 = q_index_near(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z,
                                                t.mesh[0], t.mesh[1], t.mesh[2]);
                    const int tri = tri_code_sampled(a, ch, m0, q1, q2, q3, N);
                    if (tri < 0) continue;
                    acc_cev += NB * NB * NB;                     // this q'' is visited
                    // |Δ32| of every pair lies in [b + min ω'' - max ω''', b + max ω'' - min ω''']
                    // (FP32 sums are monotonic)
                    const float4 r2 = t.wrange[q2], r3 = t.wrange[q3];
                    const float lo2 = s2 > 0 ? r2.x : -r2.y, hi2 = s2 > 0 ? r2.y : -r2.x;
                    const float thr = ADA ? fmaf(wide, r2.z + r3.z, a.ad_e0) : a.hi32;
                    unsigned near = 0;
#pragma unroll
                    for (int j1 = 0; j1 < NB; ++j1)
                        if (((base32[j1] + lo2) - r3.y) <= thr && ((base32[j1] + hi2) - r3.x) >= -thr) near |= 1u << j1;
                    near &= vm1;
                    if (!near) continue;
                    float w2f[NB], w3f[NB];
#pragma unroll
                    for (int j = 0; j < NB; ++j) {
                        w2f[j] = (float)s2 * t.omT32[j * N + q2];   // branch-major: lanes read consecutive q
                        w3f[j] = t.omT32[j * N + q3];
                    }
                    float T2[NB], T3[NB];                            // a pair's window is at most T2 + T3
#pragma unroll
                    for (int j = 0; j < NB; ++j) {
                        T2[j] = ADA ? fmaf(wide, t.pnT32[j * N + q2], a.ad_e0) : 0.0f;
                        T3[j] = ADA ? wide * t.pnT32[j * N + q3] : 0.0f;
                    }
#pragma unroll 1
                    for (int j1 = 0; j1 < NB; ++j1) {
                        if (!((near >> j1) & 1u)) continue;
                        const float b1 = w0f + (float)s1 * t.om32[q1 * NB + j1];
                        float mn = __int_as_float(0x7f800000);
#pragma unroll
                        for (int j2 = 0; j2 < NB; ++j2) {
                            const float t2 = b1 + w2f[j2];
                            float r = fabsf(t2 - w3f[0]) - T3[0];     // six short chains
#pragma unroll
                            for (int j3 = 1; j3 < NB; ++j3) r = fminf(r, fabsf(t2 - w3f[j3]) - T3[j3]);
                            mn = fminf(mn, r - T2[j2]);
                        }
                        if (!(mn <= (ADA ? 0.0f : thr))) near &= ~(1u << j1);
                    }
                    cand[k] = near | ((unsigned)tri << 8);
                    n_cand += __popc(near);
                }
                int n_all, co = block_exclusive_scan(n_cand, s_scan, &n_all);
#pragma unroll
                for (int k = 0; k < kQPT; ++k)
                    for (unsigned m = cand[k] & 0xffu; m; m &= m - 1)
                        sC[co++] = ((unsigned)(k * kTileQ + threadIdx.x) << 16) | ((unsigned)(__ffs(m) - 1) << 8) |
                                   (cand[k] >> 8);
                __syncthreads();
                total = 0;
                for (int cf = 0; cf < n_all; cf += kTileQ) {
                    unsigned long long e = 0;
                    if (cf + (int)threadIdx.x < n_all) {
                        const unsigned cw = sC[cf + threadIdx.x];
                        const int ixr = (int)(cw >> 16), j1 = (int)((cw >> 8) & 0xffu), tri = (int)(cw & 0xffu);
                        const int q2 = cb + qb + ixr;
                        const int4 c2 = t.qc[q2];
                        const int q3 = q_index_near(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z,
                                                    t.mesh[0], t.mesh[1], t.mesh[2]);
                        const unsigned v2 = t.vmask[q2], v3 = t.vmask[q3];
                        const float b = w0f + (float)s1 * t.om32[q1 * NB + j1];
                        unsigned long long near = 0, okm = 0, keep = 0;
                        float t2[NB], T2[NB];
#pragma unroll
                        for (int j2 = 0; j2 < NB; ++j2) {
                            t2[j2] = b + (float)s2 * t.om32[q2 * NB + j2];
                            T2[j2] = ADA ? fmaf(wide, t.pnT32[j2 * N + q2], a.ad_e0) : a.hi32;
                        }
                        unsigned row = v2 & ((1u << NB) - 1u);
                        if (tri == 3) row &= ~((1u << j1) - 1u);             // j'' >= j'
#pragma unroll
                        for (int j3 = 0; j3 < NB; ++j3) {
                            const float w3 = t.om32[q3 * NB + j3], T3 = ADA ? wide * t.pnT32[j3 * N + q3] : 0.0f;
                            if ((v3 >> j3) & 1u) okm |= (unsigned long long)row << (NB * j3);
#pragma unroll
                            for (int j2 = 0; j2 < NB; ++j2)
                                near |= (unsigned long long)((ADA ? fabsf(t2[j2] - w3) - T3 : fabsf(t2[j2] - w3)) <= T2[j2])
                                        << (NB * j3 + j2);
                        }
                        near &= okm;
                        while (near) {                           // the few pairs within reach, one by one
                            const int k = __ffsll(near) - 1;
                            near &= near - 1;
                            const int j3 = k / NB, j2 = k - j3 * NB;
                            const int m2 = q2 * NB + j2, m3 = q3 * NB + j3;
                            const float ad = fabsf((b + (float)s2 * t.om32[m2]) - t.om32[m3]);
                            bool kp;
                            if constexpr (ADA) {
                                const int w = window_adaptive32(a, ad, two_sigma32(t, a, m2, m3));
                                kp = w == 2 || (w == 1 && window_exact_adaptive(t, a, ch, m0, q1 * NB + j1, m2, m3, m2, m3));
                            } else {
                                kp = ad <= a.lo32 || window_exact4(ch, w0, t.om[q1 * NB + j1], t.om[m2], t.om[m3], a.two_sigma);
                            }
                            keep |= (unsigned long long)kp << k;
                        }
                        if (keep) e = ((unsigned long long)ixr << 48) | ((unsigned long long)j1 << 40) |
                                      ((unsigned long long)tri << 36) | keep;
                    }
                    const unsigned bal = __ballot_sync(kFull, e != 0);
                    if ((threadIdx.x & 31) == 0) s_scan[threadIdx.x >> 5] = __popc(bal);
                    __syncthreads();
                    int o = total + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u));
#pragma unroll
                    for (int w = 0; w < kTileQ / 32; ++w) {
                        if (w < (int)(threadIdx.x >> 5)) o += s_scan[w];
                        total += s_scan[w];
                    }
                    if (e) sQ[o] = e;
                    __syncthreads();
                }
            } else {
            // window: this thread's q'' of the round (up to kQPT) against every partner branch j'
            unsigned long long ent[NB * kQPT];
            for (int ix = qb + threadIdx.x; ix < min(cnt, qb + kTileQ * kQPT); ix += kTileQ) {
                const int q2 = cb + (pm_list ? (int)s_tri[ix] : ix);
                const int4 c2 = t.qc[q2];
                const int q3 = q_index_near(b0 + s2 * c2.x, b1 + s2 * c2.y, b2 + s2 * c2.z,
                                            t.mesh[0], t.mesh[1], t.mesh[2]);
                const unsigned v2 = t.vmask[q2], v3 = t.vmask[q3];
                float w2f[NB], w3f[NB];
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    w2f[j] = (float)s2 * t.omT32[j * N + q2];   // branch-major: lanes read consecutive q
                    w3f[j] = t.omT32[j * N + q3];
                }
                // Triangular domain (partner-swap symmetry of the summand): +- is symmetric under
                // (λ'', λ''') (q'' <-> q''' at fixed q'), ++ and -- under (λ', λ'') (q' <-> q'') when σ
                // is fixed.  One representative of each pair is evaluated with weight 2; a self-paired
                // point keeps the ordered half of its branch pairs.  The exact window test and the
                // summand are swap-symmetric, so counts and Γ equal those of the rectangular sum.
                // 0: weight 1; 1: weight 2; 2: +- with q'' = q'''; 3: ++/-- with q'' = q'; -1: the
                // swap of a pair evaluated elsewhere, or (sampling estimate) a pair outside the sample
                const int tri = tri_code_sampled(a, ch, m0, q1, q2, q3, N);
                if (tri < 0) continue;
                acc_cev += NB * NB * NB;                         // this q'' is visited
                // (j'', j''') pairs whose two partners both take part: bit NB j''' + j''
                unsigned long long okm = 0;
#pragma unroll
                for (int j3 = 0; j3 < NB; ++j3)
                    if ((v3 >> j3) & 1u) {
                        unsigned row = v2 & ((1u << NB) - 1u);
                        if (tri == 2) row &= (2u << j3) - 1u;    // j'' <= j'''
                        okm |= (unsigned long long)row << (NB * j3);
                    }
                // Adaptive ++, --: |Δ32| of every pair lies in [b + min ω'' - max ω''', b + max ω'' - min ω''']
                // (FP32 sums are monotonic), and no width exceeds the one of |P''| + |P'''|: most q'' need none.
                unsigned j1_near = vm1;
                if constexpr (ADA) {
                    if (ch != 3) {
                        const float4 r2 = t.wrange[q2], r3 = t.wrange[q3];
                        const float lo2 = s2 > 0 ? r2.x : -r2.y, hi2 = s2 > 0 ? r2.y : -r2.x;
                        const float thr = fmaf(a.ad_rhi, a.ad_c32 * (r2.z + r3.z), a.ad_e0);
#pragma unroll
                        for (int j1 = 0; j1 < NB; ++j1)
                            if (!(((base32[j1] + lo2) - r3.y) <= thr && ((base32[j1] + hi2) - r3.x) >= -thr))
                                j1_near &= ~(1u << j1);
                        if (!j1_near) continue;
                    }
                }
                // Adaptive σ: the width of a pair (λ'', λ''') does not depend on j', so the 36 widths
                // of this q'' are formed once, kept in this thread's column of s_g, and tested below
                // against every j' (branch-free masks as for a fixed σ, rare exact decisions out of line).
                if constexpr (ADA) {
#pragma unroll 1
                    for (int j3 = 0; j3 < NB; ++j3) {
                        const float4 h3 = t.vpT32[j3 * N + q3], l3 = t.vpTlo[j3 * N + q3];
#pragma unroll
                        for (int j2 = 0; j2 < NB; ++j2)
                            s_g[(j3 * NB + j2) * kTileQ + threadIdx.x] =
                                a.ad_c32 * vel_diff_norm32_approx(t.vpT32[j2 * N + q2], t.vpTlo[j2 * N + q2], h3, l3);
                    }
                }
                // Adaptive ++, --: most (q'', j') have no pair near its window at all.  The necessary
                // condition min over (j'', j''') of |Δ32| - (r_hi 2σ32 + e0) <= 0 is evaluated for all
                // j' at once, so each width is read and scaled once per q'' instead of once per j'.
                if constexpr (ADA) {
                    if (ch != 3) {
                        float mn[NB];
#pragma unroll
                        for (int j1 = 0; j1 < NB; ++j1) mn[j1] = 1.0f;
#pragma unroll
                        for (int j2 = 0; j2 < NB; ++j2) {
                            float th[NB];
#pragma unroll
                            for (int j3 = 0; j3 < NB; ++j3)
                                th[j3] = fmaf(a.ad_rhi, s_g[(j3 * NB + j2) * kTileQ + threadIdx.x], a.ad_e0);
#pragma unroll
                            for (int j1 = 0; j1 < NB; ++j1) {
                                const float t2 = base32[j1] + w2f[j2];
#pragma unroll
                                for (int j3 = 0; j3 < NB; ++j3) mn[j1] = fminf(mn[j1], fabsf(t2 - w3f[j3]) - th[j3]);
                            }
                        }
#pragma unroll
                        for (int j1 = 0; j1 < NB; ++j1)
                            if (!(mn[j1] <= 0.0f)) j1_near &= ~(1u << j1);
                    }
                }
#pragma unroll 1
                for (int j1 = 0; j1 < NB; ++j1) {
                    if (!((j1_near >> j1) & 1u)) continue;
                    const float b = base32[j1];
                    unsigned long long okj = okm;                // tri 3: j'' >= j'
                    if (tri == 3) {
                        const unsigned long long row = (unsigned long long)(((1u << NB) - 1u) & ~((1u << j1) - 1u));
                        unsigned long long cm = 0;
#pragma unroll
                        for (int j3 = 0; j3 < NB; ++j3) cm |= row << (NB * j3);
                        okj &= cm;
                    }
                    const unsigned long long tri_bits = (unsigned long long)tri << 36;
                    if constexpr (ADA) {
                        unsigned long long sure = 0, amb = 0;
#pragma unroll
                        for (int j3 = 0; j3 < NB; ++j3)
#pragma unroll
                            for (int j2 = 0; j2 < NB; ++j2) {
                                const float g = s_g[(j3 * NB + j2) * kTileQ + threadIdx.x];
                                const float ad = fabsf((b + w2f[j2]) - w3f[j3]);
                                const int k = NB * j3 + j2;
                                sure |= (unsigned long long)(ad <= fmaf(a.ad_rlo, g, -a.ad_e0) && g > a.ad_gmin) << k;
                                amb |= (unsigned long long)(ad <= fmaf(a.ad_rhi, g, a.ad_e0)) << k;
                            }
                        sure &= okj;
                        amb &= okj & ~sure;
                        while (amb) {                            // rare: exact FP64 σ and Δ
                            const int k = __ffsll(amb) - 1;
                            amb &= amb - 1;
                            const int j3 = k / NB, j2 = k - j3 * NB;
                            if (window_exact_adaptive(t, a, ch, m0, q1 * NB + j1, q2 * NB + j2, q3 * NB + j3,
                                                      q2 * NB + j2, q3 * NB + j3))
                                sure |= 1ull << k;
                        }
                        if (sure)
                            ent[n_ent++] = ((unsigned long long)(ix - qb) << 48) |
                                           ((unsigned long long)j1 << 40) | tri_bits | sure;
                        continue;
                    }
                    float t2[NB];
#pragma unroll
                    for (int j2 = 0; j2 < NB; ++j2) t2[j2] = b + w2f[j2];
                    if (ch != 3) {       // ++, --: most (q'', j') have no pair near the window at all
                        float mn = fabsf(t2[0] - w3f[0]);
#pragma unroll
                        for (int j3 = 0; j3 < NB; ++j3)
#pragma unroll
                            for (int j2 = 0; j2 < NB; ++j2) mn = fminf(mn, fabsf(t2[j2] - w3f[j3]));
                        if (!(mn <= a.hi32)) continue;          // nothing kept, nothing ambiguous
                    }
                    unsigned long long le_lo = 0, le_hi = 0;    // |Δ32| <= lo32, |Δ32| <= hi32
#pragma unroll
                    for (int j3 = 0; j3 < NB; ++j3)
#pragma unroll
                        for (int j2 = 0; j2 < NB; ++j2) {
                            const float ad = fabsf(t2[j2] - w3f[j3]);
                            le_lo |= (unsigned long long)(ad <= a.lo32) << (NB * j3 + j2);
                            le_hi |= (unsigned long long)(ad <= a.hi32) << (NB * j3 + j2);
                        }
                    unsigned long long sure = le_lo & okj, amb = le_hi & ~le_lo & okj;
                    while (amb) {                                // rare: exact FP64 decision
                        const int k = __ffsll(amb) - 1;
                        amb &= amb - 1;
                        const int j3 = k / NB, j2 = k - j3 * NB;
                        if (window_exact4(ch, w0, t.om[q1 * NB + j1], t.om[q2 * NB + j2], t.om[q3 * NB + j3],
                                          a.two_sigma))
                            sure |= 1ull << k;
                    }
                    if (sure)
                        ent[n_ent++] = ((unsigned long long)(ix - qb) << 48) |
                                       ((unsigned long long)j1 << 40) | tri_bits | sure;
                }
            }
            off = block_exclusive_scan(n_ent, s_scan, &total);
            for (int k = 0; k < n_ent; ++k) sQ[off + k] = ent[k];
            __syncthreads();
            }

            // Compacted: the block's entries are dealt out to the threads in order.
            // FP64: 32 to a warp at a time.  A lane forms its entry's X; the warp then takes the items
            // (q'', j', j''') of its 32 entries one per lane (X by shuffles from the entry's lane) and the
            // processes of 32 items one per lane (Y by shuffles), since entries carry 1-6 items and items
            // 1-6 processes, and an idle lane costs the FP64 pipe as much as a busy one.  The weights
            // return through shared memory to the lane that owns the entry, which adds them in the
            // entry's order (4 q points of 8^3: 61.5 -> 52 ms for the three channels; 43 with mirror keys
            // paired).
            // FP32: each thread walks its entry's items and processes.  Redistributed as above it was
            // slower (+- of 8^3 314 -> 414 ms; processes only, 16^3: 102 -> 132 ms): shuffles and scans
            // lengthen the chain of each warp, and 3-4 warps per scheduler do not cover it.
            // The ablation instantiation (NOCOMP, fc4_set_ablation) has each thread evaluate the entries
            // its own window found, as an uncompacted GPU-only loop would.
            if constexpr (WARP) {
              if (total && !have_w) {
                for (int k = threadIdx.x; k < NB * nk * 9; k += kTileQ) {
                    const int j = k / (nk * 9), rem = k - j * (nk * 9);
                    sW[k] = paired_value(t.perm4, rem / 9, src + j * (nk * 9) + rem % 9, 9);
                }
                __syncthreads();
                have_w = true;
              }
              const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
              unsigned char *wItem = s_item + wid * 32 * NB;
              unsigned char *wProc = s_proc + wid * 32 * NB;
              R *wVal = s_val + wid * 32 * NB * NV;
              for (int ib = wid * 32; ib < total; ib += kTileQ) {
                unsigned long long e = 0;
                int iq2 = 0, iq3 = 0;
                C X[NA][NA][9];
                if (ib + lane < total) {
                    ++acc_ent;
                    e = sQ[ib + lane];
                    const int ixe = qb + (int)(e >> 48), j1 = (int)((e >> 40) & 0xff);
                    iq2 = cb + (pm_list ? (int)s_tri[ixe] : ixe);
                    const int4 cc2 = t.qc[iq2];
                    iq3 = q_index_near(b0 + s2 * cc2.x, b1 + s2 * cc2.y, b2 + s2 * cc2.z,
                                       t.mesh[0], t.mesh[1], t.mesh[2]);
                    const C *Prow = P4 + (size_t)iq2 * nk;
                    const C *Wj = sW + j1 * nk * 9;
#pragma unroll
                    for (int c = 0; c < NA; ++c)
#pragma unroll
                        for (int d = 0; d < NA; ++d)
                            paired_sum(t.perm4, t.grp_start[c * NA + d], t.pairs4[c * NA + d], t.grp_start[c * NA + d + 1], Prow, Wj,
                                       (R)s2, X[c][d]);
                }
                unsigned rows = 0;
#pragma unroll
                for (int j3 = 0; j3 < NB; ++j3)
                    if ((e >> (NB * j3)) & ((1u << NB) - 1u)) rows |= 1u << j3;
                const int n_it = __popc(rows);
                const int io = warp_exclusive_scan(n_it), n_items = __shfl_sync(kFull, io + n_it, 31);
                {
                    int o = io;
                    for (unsigned r = rows; r; r &= r - 1) wItem[o++] = (unsigned char)((lane << 3) | (__ffs(r) - 1));
                }
                __syncwarp();
                for (int ip = 0; ip < n_items; ip += 32) {
                    const bool act = ip + lane < n_items;
                    const int code = act ? wItem[ip + lane] : 0;
                    const int src = code >> 3, j3 = code & 7;
                    const unsigned long long es = __shfl_sync(kFull, e, src);
                    const int sq2 = __shfl_sync(kFull, iq2, src), sq3 = __shfl_sync(kFull, iq3, src);
                    const unsigned m = act ? (unsigned)(es >> (NB * j3)) & ((1u << NB) - 1u) : 0u;
                    if (act) ++acc_items;
                    C Y[NA][3];
#pragma unroll
                    for (int c = 0; c < NA; ++c)
#pragma unroll
                        for (int g = 0; g < 3; ++g) Y[c][g] = czero<C>();
#pragma unroll
                    for (int d = 0; d < NA; ++d) {
                        C e3[3];
#pragma unroll
                        for (int dl = 0; dl < 3; ++dl) e3[dl] = cconj(ev[(sq3 * NB + 3 * d + dl) * NB + j3]);
#pragma unroll
                        for (int c = 0; c < NA; ++c)
#pragma unroll
                            for (int g = 0; g < 3; ++g)
#pragma unroll
                                for (int dl = 0; dl < 3; ++dl)
                                    Y[c][g] = cfma(cshfl(X[c][d][3 * g + dl], src), e3[dl], Y[c][g]);
                    }
                    const int np = __popc(m);
                    const int po = warp_exclusive_scan(np), n_proc = __shfl_sync(kFull, po + np, 31);
                    {
                        int o = po;
                        for (unsigned mm = m; mm; mm &= mm - 1) wProc[o++] = (unsigned char)((lane << 3) | (__ffs(mm) - 1));
                    }
                    // processes of this lane's own entry in the pass
                    const int lo = max(io, ip) - ip, hi = min(io + n_it, ip + 32) - ip;
                    const int from = __shfl_sync(kFull, po, lo & 31);
                    const int end = __shfl_sync(kFull, po + np, (hi - 1) & 31), to = lo < hi ? end : from;
                    // j', j''' and the domain code of the item
                    const int jj = (int)((es >> 40) & 0xff) | (j3 << 8) | ((int)((es >> 36) & 3u) << 16);
                    __syncwarp();
                    for (int pp = 0; pp < n_proc; pp += 32) {
                        const bool pact = pp + lane < n_proc;
                        const int pc = pact ? wProc[pp + lane] : 0;
                        const int il = pc >> 3, j2 = pc & 7;
                        const int pjj = __shfl_sync(kFull, jj, il);
                        const int j1 = pjj & 0xff, pj3 = (pjj >> 8) & 0xff, tri = pjj >> 16;
                        const int m1 = q1 * NB + j1;
                        const int m2 = __shfl_sync(kFull, sq2, il) * NB + j2, m3 = __shfl_sync(kFull, sq3, il) * NB + pj3;
                        const C *e2p = ev + (size_t)(m2 - j2) * NB + j2;
                        C V = czero<C>();
#pragma unroll
                        for (int c = 0; c < NA; ++c)
#pragma unroll
                            for (int g = 0; g < 3; ++g)
                                V = cfma(cconj_if(e2p[(3 * c + g) * NB], s2 < 0), cshfl(Y[c][g], il), V);
                        const double d = delta_exact(ch, w0, t.om[m1], t.om[m2], t.om[m3]);
                        double g;
                        if constexpr (ADA) g = gauss_adaptive(t, a, d, m2, m3);
                        else g = exp(-(d * d) * a.inv_sigma2) * a.gnorm;
                        R w = sym4<double>(ch) * occupation_factor<double>(ch, occ[m1], occ[m2], occ[m3]) *
                              g * invw[m0] * invw[m1] * invw[m2] * invw[m3];
                        const int wt = tri_weight(tri, j1, j2, pj3);
                        w *= (R)wt;
                        if (pact) {
                            R *v = wVal + (pp + lane) * NV;
                            v[0] = w;
                            v[1] = V.x * V.x + V.y * V.y;
                            acc_n += wt;
                            acc_ev += 1;
                            if constexpr (BTE) {
                                const R *F = Sel<R>::bteF(a);
                                const R o1 = (R)(ch == 4 ? 1 : -1) * Sel<R>::om(t)[m1];
                                const R o2 = (R)(ch == 2 ? -1 : 1) * Sel<R>::om(t)[m2];
                                const R o3 = Sel<R>::om(t)[m3];
#pragma unroll
                                for (int x = 0; x < 3; ++x)
                                    v[2 + x] = (o1 * F[3 * m1 + x] + o2 * F[3 * m2 + x]) + o3 * F[3 * m3 + x];
                            }
                        }
                    }
                    __syncwarp();
                    for (int k = from; k < to; ++k) {
                        const R *v = wVal + k * NV;
                        acc_wp.add(v[0]);
                        acc_g.add(v[0] * v[1]);
                        if constexpr (BTE) {
                            const R g = v[0] * v[1];
#pragma unroll
                            for (int x = 0; x < 3; ++x) acc_d[x].add(g * v[2 + x]);
                        }
                    }
                    __syncwarp();                                // lists reused by the next pass
                }
              }
            } else {
            for (int it = NOCOMP ? off : (int)threadIdx.x; it < (NOCOMP ? off + n_ent : total); it += NOCOMP ? 1 : kTileQ) {
                ++acc_ent;
                const unsigned long long e = sQ[it];
                const int ixe = qb + (int)(e >> 48), j1 = (int)((e >> 40) & 0xff);
                const int iq2 = cb + (pm_list ? (int)s_tri[ixe] : ixe);
                const int tri = (int)((e >> 36) & 3u);
                const int4 cc2 = t.qc[iq2];
                const int iq3 = q_index_near(b0 + s2 * cc2.x, b1 + s2 * cc2.y, b2 + s2 * cc2.z,
                                             t.mesh[0], t.mesh[1], t.mesh[2]);
                const int m1 = q1 * NB + j1;
                // per-entry constants of the mixed weight: TwoSum of ω + s1 ω', the sum of their lo
                // parts, n', 1/(ω ω')
                const float4 k0 = t.mode4[m0], k1 = t.mode4[m1];
                float ee1;
                const float ex1 = two_sum(k0.x, (float)s1 * k1.x, ee1);
                const float el01 = k0.y + (float)s1 * k1.y, iw01 = k0.w * k1.w, n1f = k1.z;
                const C *Prow = P4 + (size_t)iq2 * nk;
                const C *Wj = sW + j1 * nk * 9;
                C X[NA][NA][9];
#pragma unroll
                for (int c = 0; c < NA; ++c)
#pragma unroll
                    for (int d = 0; d < NA; ++d) {
#pragma unroll
                        for (int k = 0; k < 9; ++k) X[c][d][k] = czero<C>();
                        const int r0 = t.grp_start[c * NA + d], r1 = t.grp_start[c * NA + d + 1];
#pragma unroll 2
                        for (int r = r0; r < r1; ++r) {
                            const C ph = cconj_if(Prow[r], s2 < 0);
                            const C *Wr = Wj + 9 * r;
#pragma unroll
                            for (int k = 0; k < 9; ++k) X[c][d][k] = cfma(ph, Wr[k], X[c][d][k]);
                        }
                    }
                // each lane goes through its own items: the warp takes as many steps as the entry with the most
                // items has, not one per j''' that any entry has
                unsigned rows = 0;
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
#pragma unroll
                    for (int d = 0; d < NA; ++d) {
                        C e3[3];
#pragma unroll
                        for (int dl = 0; dl < 3; ++dl) e3[dl] = cconj(ev[(iq3 * NB + 3 * d + dl) * NB + j3]);
#pragma unroll
                        for (int c = 0; c < NA; ++c)
#pragma unroll
                            for (int g = 0; g < 3; ++g)
#pragma unroll
                                for (int dl = 0; dl < 3; ++dl) Y[c][g] = cfma(X[c][d][3 * g + dl], e3[dl], Y[c][g]);
                    }
                    const int m3 = iq3 * NB + j3;
                    const float4 k3 = t.mode4[m3];
                    while (m) {
                        const int j2 = __ffs(m) - 1;
                        m &= m - 1;
                        const int m2 = iq2 * NB + j2;
                        C V = czero<C>();
#pragma unroll
                        for (int c = 0; c < NA; ++c)
#pragma unroll
                            for (int g = 0; g < 3; ++g)
                                V = cfma(cconj_if(ev[(iq2 * NB + 3 * c + g) * NB + j2], s2 < 0), Y[c][g], V);
                        // Δ from the entry's TwoSum (ex1, ee1) and the hi/lo splits of the last two ω
                        float e2s, e3s;
                        const float4 k2 = t.mode4[m2];
                        const float x2 = two_sum(ex1, (float)s2 * k2.x, e2s);
                        const float x3 = two_sum(x2, -k3.x, e3s);
                        const float lo = (el01 + (float)s2 * k2.y) - k3.y;
                        const float df = x3 + ((ee1 + e2s) + (e3s + lo));
                        float gs;
                        if constexpr (ADA) gs = gauss_adaptive32(t, a, df, m2, m3);
                        else gs = __expf(-(df * df) * a.inv_sigma2_32) * a.gnorm32;
                        R w = sym4<float>(ch) * occupation_factor<float>(ch, n1f, k2.z, k3.z) * gs *
                            iw01 * (k2.w * k3.w);
                        // weight of the representative: 2 for a swapped pair, 1 on the diagonal
                        const int wt = tri_weight(tri, j1, j2, j3);
                        w *= (R)wt;
                        acc_wp.add(w);
                        acc_g.add(w * (V.x * V.x + V.y * V.y));
                        acc_n += wt;
                        acc_ev += 1;
                        if constexpr (BTE) {
                            const R *F = Sel<R>::bteF(a);
                            const R g = w * (V.x * V.x + V.y * V.y);
                            const R o1 = (R)(ch == 4 ? 1 : -1) * Sel<R>::om(t)[m1];
                            const R o2 = (R)(ch == 2 ? -1 : 1) * Sel<R>::om(t)[m2];
                            const R o3 = Sel<R>::om(t)[m3];
#pragma unroll
                            for (int x = 0; x < 3; ++x)
                                acc_d[x].add(g * ((o1 * F[3 * m1 + x] + o2 * F[3 * m2 + x]) + o3 * F[3 * m3 + x]));
                        }
                    }
                }
            }
            }
            __syncthreads();                                     // sQ reused by the next round
          }
        }
    }
    double sums[BTE ? 5 : 2];
    sums[0] = acc_g.value();
    sums[1] = acc_wp.value();
    if constexpr (BTE) {
#pragma unroll
        for (int x = 0; x < 3; ++x) sums[2 + x] = acc_d[x].value();
    }
    long long cnts[5] = {acc_n, acc_items, acc_ent, acc_ev, acc_cev};
    block_sum_multi<BTE ? 5 : 2, 5>(sums, cnts, s_red, s_redn);
    if (threadIdx.x == 0) {
        const size_t o = ((size_t)ch * a.n_modes + ms) * N + q1;
        if constexpr (BTE) {
            const double iw0 = t.invw[m0];                      // ξ_k = ω_k / ω_λ
#pragma unroll
            for (int x = 0; x < 3; ++x) a.part_d[3 * o + x] = sums[2 + x] * iw0;
        }
        a.part_g[o] = sums[0];
        a.part_wp[o] = sums[1];
        a.part_n[o] = cnts[0];
        a.part_items[o] = cnts[1];
        a.part_ent[o] = cnts[2];
        if (a.part_ev) a.part_ev[o] = cnts[3];
        if (a.part_cev) a.part_cev[o] = cnts[4];
    }
}

template <typename R, int NA>
size_t tile_smem_bytes(const Tables &t, int qpt = kQPTSparse, bool adaptive = true) {
    using C = Cplx<R>;
    constexpr int NB = 3 * NA;
    size_t b = sizeof(C) * ((size_t)NB * t.n_keys * 9) + sizeof(unsigned long long) * (size_t)kTileQ * NB * qpt +
               (adaptive ? sizeof(float) * (size_t)NB * NB * kTileQ : 0);
    return (b + 15) & ~size_t(15);
}

// W bytes per mode (all q' and j') for the tiled path
template <typename R, int NA>
size_t tile_w_bytes_per_mode(const Tables &t) {
    return sizeof(Cplx<R>) * (size_t)t.N * 3 * NA * t.n_keys * 9;
}

// Shared memory of w4_kernel.
template <typename R, int NA>
size_t w4_smem_bytes(const Tables &t) {
    constexpr int NB = 3 * NA;
    return sizeof(Cplx<R>) * ((size_t)t.nc4 * 28 + NB * NB + NB + (size_t)t.n_keys * NA * 27);
}
constexpr size_t kW4MostSmem = 227 * 1024;

// W of the units of modes [m, m + nm) into a.wbuf.  FP32 by columns where its tables fit: 240 bytes a cluster and 4 a
// (key, atom), against 224 and 216 for Ψ in shared memory, so lists of 969 to some 1030 clusters with few keys (36 and
// fewer) take w4_kernel.
template <typename R, int NA>
cudaError_t launch_w4(const Tables &t, const RateArgs &a, int ch, int m, int nm, cudaStream_t s) {
    using C = Cplx<R>;
    C *w = reinterpret_cast<C *>(a.wbuf);
    cudaError_t e;
    if (sizeof(R) == 8 || W4Smem<NA>::bytes(t) > kW4MostSmem) {
        const size_t smem = w4_smem_bytes<R, NA>(t);
        e = cudaFuncSetAttribute(w4_kernel<R, NA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const long long ngrp = (t.N + kW4Group - 1) / kW4Group;
        w4_kernel<R, NA><<<(unsigned)(nm * ngrp), kW4Threads, smem, s>>>(t, a, ch, m, w);
    } else if constexpr (sizeof(R) == 4) {
        const size_t smem = W4Smem<NA>::bytes(t);
        e = cudaFuncSetAttribute(w4_column_kernel<NA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        // q' per block: up to 32 share a Φ~ as long as the grid still fills the device
        int group = 32;
        while (group > 4 && (long long)nm * ((t.N + group - 1) / group) < 1216) group /= 2;
        const long long ngrp = (t.N + group - 1) / group;
        const int cols = t.n_keys * 9, rounds = std::max(1, (cols + 383) / 384);
        const int threads = std::max(32, ((cols + rounds - 1) / rounds + 31) / 32 * 32);
        w4_column_kernel<NA><<<(unsigned)(nm * ngrp), threads, smem, s>>>(t, a, ch, m, group, w);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess && a.n_kernels) ++*a.n_kernels;
    return e;
}

// Launch W (global) then the tiled kernel, over mode chunks that fit in the W buffer.
template <typename R, int NA, bool ADA, bool BTE = false>
cudaError_t launch4_tile(const Tables &t, const RateArgs &a, int ch, cudaStream_t s) {
    using C = Cplx<R>;
    const bool dense = ch == 3;
    const size_t smem = tile_smem_bytes<R, NA>(t, qpt_of<ADA>(dense), ADA && (dense || a.no_compact));
    auto kern = dense ? rates4_tile_kernel<R, NA, ADA, qpt_of<ADA>(true), BTE>
                      : rates4_tile_kernel<R, NA, ADA, qpt_of<ADA>(false), BTE>;
    if constexpr (sizeof(R) == 4 && !BTE)       // ablation switch: mixed precision only
        if (a.no_compact)
            kern = dense ? rates4_tile_kernel<R, NA, ADA, qpt_of<ADA>(true), false, true>
                         : rates4_tile_kernel<R, NA, ADA, qpt_of<ADA>(false), false, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const size_t per_mode = tile_w_bytes_per_mode<R, NA>(t);
    const int chunk = (int)(a.wbuf_bytes / per_mode);
    if (chunk < 1) return cudaErrorInvalidValue;
    for (int m = 0; m < a.n_modes; m += chunk) {
        const int nm = min(chunk, a.n_modes - m);
        if (!(a.w_reuse && nm == a.n_modes)) {           // W of the previous channel with the same s1
            e = launch_w4<R, NA>(t, a, ch, m, nm, s);
            if (e != cudaSuccess) return e;
        }
        if constexpr (sizeof(R) == 4 && !BTE) {
            if (ch == 3 && a.use_tc) {                  // +-: cluster contraction on the tensor cores
                e = launch_rates4_tc(t, a, ch, m, nm, reinterpret_cast<const float2 *>(a.wbuf), s);
                if (e != cudaSuccess) return e;
                if (a.n_kernels) ++*a.n_kernels;
                continue;
            }
        }
        kern<<<(unsigned)((long long)nm * t.N), kTileQ, smem, s>>>(t, a, ch, m, reinterpret_cast<const C *>(a.wbuf));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (a.n_kernels) ++*a.n_kernels;
    }
    return cudaSuccess;
}

}  // namespace fc4
