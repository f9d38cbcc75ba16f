// The online ensemble as two sweeps over the logits: what sd_sweep.cuh does for the step, with several drafts to a
// target row.  The units are positions (sequence, row); a block takes one item of a position -- some of its sampling
// regions -- of the target and of up to kEnsembleGroup drafts at once, so that a target entry is read and its
// exponential taken once for all of them, in either sweep.
//
//   sd_ensemble_stats_kernel  softmax sums of every item and learner to the workspace
//   sd_ensemble_rows_kernel   a warp to a position and learner: its items merged, row constants, loss
//   sd_ensemble_grad_kernel   the gradients; its first block does the round's losses and weights meanwhile
//
// What bounds it: HBM, where every logit is read twice but for the 80 MiB that L2 keeps.  3 learners, 32 sequences, 8
// tokens, 128 256 bf16 entries 122 us (at the copy bandwidth: 70 us for every logit once, 98 for what is moved), 144 on
// the cluster kernel, which takes the learners one after the other and the target's exponentials with each.  A group of four
// learners has three blocks an SM (four spill: 158 us against 155), smaller ones four (2 learners 87, with three blocks 90).  Three
// learners spill at four blocks, too (92 bytes of stores in the first sweep, 8 in the second; at three blocks none), and are no slower for
// it, us, four blocks / three in the first sweep / in both: 256 positions of 128 256 entries 120.8 / 121.2 / 120.3, 600 of 151 936 328 / 333 /
// 331, 144 of 32 000 20.4 / 20.4 / 20.8; 6 learners 655 / 666 / 662 and 41.2 / 43.2 / 44.6.
// bf16 rows only (rule and figures: use_ensemble_sweeps, host).
#pragma once

#include "sd_sweep.cuh"

namespace sdv {

constexpr int kEnsembleGroup = 4;      // learners that share a reading of the target

struct EnsembleSweep {
    int slices, regions;               // items of a position, sampling regions of an item
    int n0;                            // learners [n0, n0 + NL) are this launch's
    PartialStats* part;                // workspace [positions][learners][slices]
    RowConst* rowc;                    // workspace [positions][learners]
    unsigned kept;                     // items, from the last one backwards, that L2 is asked to keep between the sweeps
};

// Sums of a lane relative to integer references that its warp shares: one target, NL drafts.
template <int NL> struct EnsembleState {
    float RT, RD[NL];
    float sT, sD[NL], w[NL];
    __device__ __forceinline__ void init() {
        RT = kEmptyRef;
        sT = 0.f;
#pragma unroll
        for (int n = 0; n < NL; ++n) { RD[n] = kEmptyRef; sD[n] = w[n] = 0.f; }
    }
};

// The maxima of a region raise the references; the running sums follow (exactly).
template <int DT, int NL>
__device__ __forceinline__ void ensemble_raise(const uint4 (&rt)[kRegionRows], const uint4 (&rd)[NL][kRegionRows], float c, EnsembleState<NL>& s) {
    const float nT = fmaxf(s.RT, warp_max_ref(ref_of(region_max<DT>(rt), c)));
    const float dT = nT - s.RT, f = pow2_neg_f32(-dT);
#pragma unroll
    for (int n = 0; n < NL; ++n) {
        const float nD = fmaxf(s.RD[n], warp_max_ref(ref_of(region_max<DT>(rd[n]), c)));
        const float dD = nD - s.RD[n];
        s.w[n] = s.sT > 0.f ? (s.w[n] - s.sT * (dT - dD)) * f : 0.f;
        s.sD[n] *= pow2_neg_f32(-dD);
        s.RD[n] = nD;
    }
    s.sT *= f;
    s.RT = nT;
}

// The region's sums (entries two at a time, even and odd ones apart, as LaneSums::vector_pair has them).
template <int DT, int NL, bool MASKED>
__device__ __forceinline__ void ensemble_sums(const uint4 (&rt)[kRegionRows], const uint4 (&rd)[NL][kRegionRows], float c,
                                              const EnsembleState<NL>& s, float& sT, float (&sD)[NL], float (&sW)[NL]) {
    using E = Elem<DT>;
    constexpr int VEC = E::VEC;
    const float2 c2 = make_float2(c, c), m1 = make_float2(-1.f, -1.f), nT2 = make_float2(-s.RT, -s.RT);
    sT = 0.f;
#pragma unroll
    for (int n = 0; n < NL; ++n) sD[n] = sW[n] = 0.f;
#pragma unroll
    for (int g = 0; g < kRegionRows; ++g) {
        float t[VEC];
        E::unpack(rt[g], t);
        float2 aT[VEC / 2], eT[VEC / 2], accT = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < VEC / 2; ++e) {
            aT[e] = __ffma2_rn(make_float2(t[2 * e], t[2 * e + 1]), c2, nT2);
            eT[e] = make_float2(ex2f(aT[e].x), ex2f(aT[e].y));
            accT = __fadd2_rn(accT, eT[e]);
        }
        sT += accT.x + accT.y;
#pragma unroll
        for (int n = 0; n < NL; ++n) {
            const float2 nD2 = make_float2(-s.RD[n], -s.RD[n]);
            float d[VEC];
            E::unpack(rd[n][g], d);
            float2 accD = make_float2(0.f, 0.f), accW = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < VEC / 2; ++e) {
                const float2 aD = __ffma2_rn(make_float2(d[2 * e], d[2 * e + 1]), c2, nD2);
                accD = __fadd2_rn(accD, make_float2(ex2f(aD.x), ex2f(aD.y)));
                const float2 diff = __ffma2_rn(aD, m1, aT[e]);               // aT - aD
                if constexpr (MASKED) {
                    if (eT[e].x > 0.f) accW.x = __fmaf_rn(eT[e].x, diff.x, accW.x);    // masked target entries (p = 0) add nothing
                    if (eT[e].y > 0.f) accW.y = __fmaf_rn(eT[e].y, diff.y, accW.y);
                } else {
                    accW = __ffma2_rn(eT[e], diff, accW);
                }
            }
            sD[n] += accD.x + accD.y;
            sW[n] += accW.x + accW.y;
        }
    }
}

template <int DT, int NL>
__device__ __forceinline__ void ensemble_load(const uint4* gT, const uint4* const (&gD)[NL], int v, int nvec, int lane, uint64_t policy,
                                              uint4 (&rt)[kRegionRows], uint4 (&rd)[NL][kRegionRows]) {
#pragma unroll
    for (int g = 0; g < kRegionRows; ++g) {
        const int vi = g * 32 + lane;
        const bool in = vi < nvec;                   // (what is behind the row's end reads as -inf)
        rt[g] = in ? load_l2(gT + v + vi, policy) : Elem<DT>::masked();
#pragma unroll
        for (int n = 0; n < NL; ++n) rd[n][g] = in ? load_l2(gD[n] + v + vi, policy) : Elem<DT>::masked();
    }
}

// A region once more, the slow way (as pass1_region_again).
template <int DT, int NL>
__device__ __noinline__ EnsembleState<NL> ensemble_region_again(const Params& P, const EnsembleSweep& S, size_t t_row, size_t d_row, int v, int nvec,
                                                                EnsembleState<NL> s) {
    using ET = typename Elem<DT>::type;
    const int lane = threadIdx.x & 31;
    const uint4* gD[NL];
#pragma unroll
    for (int n = 0; n < NL; ++n) gD[n] = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.Dn[S.n0 + n]) + d_row * P.V);
    uint4 rt[kRegionRows], rd[NL][kRegionRows];
    ensemble_load<DT, NL>(reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + t_row * P.V), gD, v, nvec, lane, policy_normal(), rt, rd);
    ensemble_raise<DT, NL>(rt, rd, P.c, s);
    float sT, sD[NL], sW[NL];
    ensemble_sums<DT, NL, true>(rt, rd, P.c, s, sT, sD, sW);
    s.sT += sT;
#pragma unroll
    for (int n = 0; n < NL; ++n) { s.sD[n] += sD[n]; s.w[n] += sW[n]; }
    return s;
}

// Position `pos` = sequence * k + row.  One block per item: blockIdx.x = position, blockIdx.y = slice.
template <int DT, int NL>
__global__ void __launch_bounds__(kSweepThreads, NL < 4 ? 4 : 3)
sd_ensemble_stats_kernel(const __grid_constant__ Params P, const __grid_constant__ EnsembleSweep S) {
    using E = Elem<DT>;
    using ET = typename E::type;
    constexpr float kTooLarge = 1.152921504606846976e18f;   // 2^60
    __shared__ PartialStats wpart[NL][kSweepWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int pos = blockIdx.x, slice = blockIdx.y, b = pos / P.k;
    const size_t t_row = (size_t)pos + b;
    await_previous_kernel();
    launch_dependents();
    if (P.status && threadIdx.x == 0 && S.n0 == 0 && slice == 0 && pos == b * P.k) P.status[b] = 0;      // (ORed in by the rows kernel)
    EnsembleState<NL> s;
    s.init();
    const unsigned from_end = (gridDim.y - 1u - blockIdx.y) * gridDim.x + (gridDim.x - 1u - blockIdx.x);
    const uint64_t policy = from_end < S.kept ? policy_keep() : policy_discard();
    const uint4* const gT = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + t_row * P.V);
    const uint4* gD[NL];
#pragma unroll
    for (int n = 0; n < NL; ++n) gD[n] = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.Dn[S.n0 + n]) + (size_t)pos * P.V);
    int v = (slice * S.regions + warp) * kRegionVecs, end = min((slice + 1) * S.regions * kRegionVecs, P.V / E::VEC);
    if (!SD_IN(t_row, (long long)P.B * (P.k + 1), 10) || !SD_IN(pos, (long long)P.B * P.k, 11) || !SD_IN((long long)end * E::VEC - 1, P.V, 10)) end = 0;
    bool first = true;
    for (; v + kRegionVecs <= end; v += kSweepStep, first = false) {
        uint4 rt[kRegionRows], rd[NL][kRegionRows];
        ensemble_load<DT, NL>(gT, gD, v, kRegionVecs, lane, policy, rt, rd);
        if (first) ensemble_raise<DT, NL>(rt, rd, P.c, s);
        float sT, sD[NL], sW[NL];
        ensemble_sums<DT, NL, false>(rt, rd, P.c, s, sT, sD, sW);
        // masked target entries (NaN) or entries far above the references: maxima first, then the sums
        bool bad = !(sT < kTooLarge);
#pragma unroll
        for (int n = 0; n < NL; ++n) bad = bad || !(sD[n] < kTooLarge) || sW[n] != sW[n];
        if (__any_sync(0xffffffffu, bad)) {
            s = ensemble_region_again<DT, NL>(P, S, t_row, pos, v, kRegionVecs, s);
            continue;
        }
        s.sT += sT;
#pragma unroll
        for (int n = 0; n < NL; ++n) { s.sD[n] += sD[n]; s.w[n] += sW[n]; }
    }
    if (v < end) s = ensemble_region_again<DT, NL>(P, S, t_row, pos, v, end - v, s);       // cut short by the end of the row
#pragma unroll
    for (int n = 0; n < NL; ++n) {
        LaneSums ls;
        ls.sT = s.sT; ls.sD = s.sD[n]; ls.w = s.w[n];
        warp_post_lanes(ls, s.RT, s.RD[n], lane, &wpart[n][warp]);
    }
    __syncthreads();
    if (warp < NL) {
        // a warp to a learner
        const PartialStats item = warp_merge_lanes(lane < kSweepWarps ? wpart[warp][lane] : empty_partial());
        const size_t row = (size_t)pos * P.learners + S.n0 + warp;
        if (lane == 0 && SD_IN(row, (long long)P.B * P.k * P.learners, 26) && SD_IN(slice, S.slices, 26)) S.part[row * S.slices + slice] = item;
    }
}

// A warp to a position and learner.
__global__ void __launch_bounds__(kSweepThreads)
sd_ensemble_rows_kernel(const __grid_constant__ Params P, const __grid_constant__ EnsembleSweep S) {
    const int lane = threadIdx.x & 31;
    const long long rows = (long long)P.B * P.k * P.learners, row = (long long)blockIdx.x * kSweepWarps + (threadIdx.x >> 5);
    launch_dependents();
    await_previous_kernel();
    if (row >= rows) return;
    const PartialStats st = warp_merge_lanes(lane < S.slices ? load_partial_cg(S.part + row * S.slices + lane) : empty_partial());
    const RowLogs logs = warp_row_logs(st);
    if (lane != 0) return;
    const long long pos = row / P.learners;
    const int n = (int)(row - pos * P.learners);
    S.rowc[row] = row_constants_of(P.inv_tau, false, st);
    const bool ok = st.sT > 0.0 && isfinite(st.sT) && st.sD > 0.0 && isfinite(st.sD);
    if (!ok && P.status) atomicOr(P.status + pos / P.k, SD_STATUS_BAD_ROW);
    P.loss[(long long)n * P.B * P.k + pos] = (float)(0.6931471805599453 * (st.w / st.sT - logs.T + logs.D));
}

// What the round comes to: mean losses, cumulative losses, Hedge weights.
struct HedgeArgs {
    double eps;
    const double* cum_in;
    double *round_loss, *cum_out;
    float* weights;
};

// Block 0: the round, a warp to a learner (S.n0 = 0).  The others: an item each, from the last one of the first sweep backwards.
template <int DT, int NL>
__global__ void __launch_bounds__(kSweepThreads, NL < 4 ? 4 : 3)
sd_ensemble_grad_kernel(const __grid_constant__ Params P, const __grid_constant__ EnsembleSweep S, const __grid_constant__ HedgeArgs H) {
    using E = Elem<DT>;
    using ET = typename E::type;
    constexpr int VEC = E::VEC;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int positions = P.B * P.k, id = (int)(gridDim.x - 1u - blockIdx.x), slice = id / positions, pos = id - slice * positions;
    await_previous_kernel();
    launch_dependents();
    if (blockIdx.x == 0) {
        if (S.n0 != 0) return;
        __shared__ double part[kMaxLearners];
        static_assert(kMaxLearners <= kSweepWarps, "a warp to a learner");
        if (warp < P.learners) hedge_sum(P.loss + (size_t)warp * positions, positions, lane, 32, part[warp]);
        __syncthreads();
        if (warp == 0) hedge_weights(P.learners, part[min(lane, P.learners - 1)] / (double)positions, H.eps, H.cum_in, H.round_loss, H.cum_out, H.weights);
        return;
    }
    if (!SD_IN(slice, S.slices, 20) || !SD_IN((long long)pos + pos / P.k, (long long)P.B * (P.k + 1), 12)) return;
    const uint4* const gT = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + ((size_t)pos + pos / P.k) * P.V);
    const uint4* gD[NL];
    uint4* gG[NL];
    RowConst rc[NL];
#pragma unroll
    for (int n = 0; n < NL; ++n) {
        rc[n] = S.rowc[(size_t)pos * P.learners + S.n0 + n];
        gD[n] = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.Dn[S.n0 + n]) + (size_t)pos * P.V);
        gG[n] = P.Gn[S.n0 + n] ? reinterpret_cast<uint4*>(reinterpret_cast<ET*>(P.Gn[S.n0 + n]) + (size_t)pos * P.V) : nullptr;
    }
    const uint64_t policy = policy_discard();
    const float2 c2 = make_float2(P.c, P.c), nT2 = make_float2(rc[0].negRT, rc[0].negRT), kT2 = make_float2(-rc[0].kT, -rc[0].kT);
    int end = min((slice + 1) * S.regions * kRegionVecs, P.V / VEC);
    if (!SD_IN((long long)end * VEC - 1, P.V, 12)) end = 0;
    for (int v = (slice * S.regions + warp) * kRegionVecs; v < end; v += kSweepStep) {
        uint4 rt[kRegionRows], rd[NL][kRegionRows];
        const int nvec = min(kRegionVecs, end - v);
        ensemble_load<DT, NL>(gT, gD, v, nvec, lane, policy, rt, rd);
#pragma unroll
        for (int g = 0; g < kRegionRows; ++g) {
            const int vi = g * 32 + lane;
            float t[VEC];
            E::unpack(rt[g], t);
            float2 pT[VEC / 2];                          // -(eT * kT)
#pragma unroll
            for (int e = 0; e < VEC / 2; ++e) {
                const float2 aT = __ffma2_rn(make_float2(t[2 * e], t[2 * e + 1]), c2, nT2);
                pT[e] = __fmul2_rn(make_float2(ex2f(aT.x), ex2f(aT.y)), kT2);
            }
#pragma unroll
            for (int n = 0; n < NL; ++n) {
                float d[VEC], gv[VEC];
                E::unpack(rd[n][g], d);
#pragma unroll
                for (int e = 0; e < VEC / 2; ++e) {
                    const float2 aD = __ffma2_rn(make_float2(d[2 * e], d[2 * e + 1]), c2, make_float2(rc[n].negRD, rc[n].negRD));
                    const float2 g2 = __ffma2_rn(make_float2(ex2f(aD.x), ex2f(aD.y)), make_float2(rc[n].kD, rc[n].kD), pT[e]);
                    gv[2 * e] = g2.x;
                    gv[2 * e + 1] = g2.y;
                }
                if (gG[n] && vi < nvec) store_streaming(gG[n] + v + vi, E::pack(gv));
            }
        }
    }
}

}  // namespace sdv
