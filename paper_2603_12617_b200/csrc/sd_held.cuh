// The step with the logits held in registers: every logit is read once, by the lane that works on it, and
// nothing is read again.  A unit (sequence, row) belongs to a cluster of C blocks; its sampling regions are
// dealt to the cluster's warps in order, at most N to a warp, and all of a warp's loads are in flight
// together.  Between the two passes the warps exchange their softmax sums through distributed shared
// memory, after the second one their masses, and the warp whose regions hold u * total searches them where
// they are.  Clusters meet only in a sequence's tickets: whoever takes the last one writes accept length
// and tokens.  The only waits are hardware barriers of a cluster.
//
// For calls whose rows are all on the chip at once (up to 19 MB of logits, 128 KiB an SM): what bounds them is the
// chain of dependent steps.  1 sequence, 4 tokens, 32 000 fp32 entries, 8.8 us a call, calls back to back (11 if the next
// call could not come in while this one goes out).  Clock stamps in one unit add up to 8.7: loads and maxima 1.4, sums 0.15,
// their exchange and merge 1.35, gradient and masses 0.55, their exchange 1.9, whose the draw is 0.6, search 0.7,
// the last ticket 1.35, the end of the sequence 0.7.  sd_stream_kernel took 16.6: it
// fills a ring that is read twice, hands sums from warp to warp, and draws by one warp at the end, from
// memory.  With more rows than fit, clusters come in rounds of 13 us that nothing overlaps, and kernels that
// stream are the faster ones (rule and figures: use_held, host).
#pragma once

#include "sd_kernels.cuh"

namespace sdv {

constexpr int kHeldWarps = 16;
constexpr int kHeldThreads = kHeldWarps * 32;
constexpr int kHeldMaxCluster = 16;
constexpr int kHeldMaxRegions = 4;                        // regions of a warp
constexpr int kHeldSlots = kHeldMaxCluster * kHeldWarps;  // warps of a cluster

// What a unit leaves for the end of its sequence: the token it would emit, and status bits that count if it does.
struct HeldCandidate { int32_t token; uint32_t flags; };

struct HeldShared {
    PartialStats part[kHeldSlots];       // written by every warp of the cluster (distributed shared memory)
    double2 mass[2][kHeldSlots];         // x: a warp's mass, y: its share of the hint error
    RowConst rc;
    PartialStats row;
};

// A vector that nothing else will read, or `v` as it is.
__device__ __forceinline__ void held_load(uint4& v, const uint4* p, bool in, uint64_t policy) {
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.ne.b32 p, %5, 0;\n\t"
                 "@p ld.global.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %6;\n\t}"
                 : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "l"(p), "r"((int)in), "l"(policy));
}

// Softmax sums of a lane's part of a region of which `nv` vectors are in the row (those behind it hold -inf, for which
// the arithmetic has no test: they are left out by their place).
template <int DT, bool MASKED>
__device__ __forceinline__ void held_sums(const uint4 (&rt)[kRegionRows], const uint4 (&rd)[kRegionRows], int nv, int lane, float c,
                                          float RT, float RD, float& sT, float& sD, float& sW) {
    using E = Elem<DT>;
    sT = sD = sW = 0.f;
#pragma unroll
    for (int g = 0; g < kRegionRows; ++g) {
        float tv[E::VEC], dv[E::VEC], pT, pD, pW;
        E::unpack(rt[g], tv);
        E::unpack(rd[g], dv);
        LaneSums::vector_pair<E::VEC, MASKED>(tv, dv, c, -RT, -RD, pT, pD, pW);
        if (g * 32 + lane < nv) { sT += pT; sD += pD; sW += pW; }
    }
}

// Merge of `n` partials in shared memory by one warp.  Every lane gets the same bits.
__device__ __forceinline__ PartialStats held_merge(const PartialStats* part, int n, int lane) {
    float RT = kEmptyRef, RD = kEmptyRef;
    for (int i = lane; i < n; i += 32) { RT = fmaxf(RT, part[i].RT); RD = fmaxf(RD, part[i].RD); }
    RT = warp_max_ref(RT);
    RD = warp_max_ref(RD);
    PartialStats r;
    r.RT = RT; r.RD = RD;
    r.sT = r.sD = r.w = 0.0;
    for (int i = lane; i < n; i += 32) {
        const PartialStats q = rescaled(part[i], RT, RD);
        r.sT += q.sT; r.sD += q.sD; r.w += q.w;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        r.sT += shfl_xor_f64(r.sT, off);
        r.sD += shfl_xor_f64(r.sD, off);
        r.w += shfl_xor_f64(r.w, off);
    }
    return r;
}

// What a sequence puts out, by one warp: accept length n, token y after it, status.  first: the lane's own draft token
// (of the first 32), asked for beforehand.
__device__ __forceinline__ void held_emit(const Params& P, int b, int n, int y, uint32_t status, int32_t first, int lane) {
    const int k = P.k;
    if (lane == 0) {
        P.accept_len[b] = n;
        if (P.status) P.status[b] = status;
        P.wstatus[b] = 0;               // ready for the next call
        P.ticket[b] = 0;
    }
    for (int i = lane; i <= k; i += 32) {
        const int32_t xi = i >= n ? -1 : i == lane ? first : P.x[b * k + i];
        if (SD_IN(b * (k + 1) + i, P.B * (k + 1), 25)) P.tokens[b * (k + 1) + i] = i == n ? y : xi;
    }
}

// End of a sequence, by the warp that took its last ticket.  Of up to 32 rows a lane each asks for everything that may
// be wanted, so that one round trip does.
__device__ __forceinline__ void held_finish(const Params& P, const HeldCandidate* cand, int b, int lane) {
    const int k = P.k;
    const int32_t first = lane < k ? P.x[b * k + lane] : -1;
    const uint32_t word = __ldcg(P.wstatus + b);
    int2 c = make_int2(0, 0);
    if (lane <= k && SD_IN(b * (k + 1) + lane, P.B * (k + 1), 20)) c = __ldcg(reinterpret_cast<const int2*>(cand + b * (k + 1) + lane));
    int n = k;
    for (int i0 = 0; i0 < k; i0 += 32) {
        const int i = i0 + lane;
        const unsigned m = __ballot_sync(0xffffffffu, i < k && __ldcg(P.accept + b * k + i) == 0);
        if (m) { n = i0 + __ffs(m) - 1; break; }
    }
    if (!SD_IN(n, k + 1, 23)) return;
    c.x = __shfl_sync(0xffffffffu, c.x, n & 31);
    c.y = __shfl_sync(0xffffffffu, c.y, n & 31);
    if (n >= 32) c = __ldcg(reinterpret_cast<const int2*>(cand + b * (k + 1) + n));
    held_emit(P, b, n, c.x, word | (uint32_t)c.y, first, lane);
}

// Inverse-CDF search inside a region held in registers: `prefix` = mass before it, `t` = target.  The vocabulary
// index (in every lane) of the first entry whose running sum exceeds t; if there is none, or with `last`, of the
// last entry that has mass, or -1.
template <int DT>
__device__ __forceinline__ int held_search(const uint4 (&rt)[kRegionRows], const uint4 (&rd)[kRegionRows], int v_first, int lane,
                                           float c, const RowConst& rc, double prefix, double t, bool last) {
    using E = Elem<DT>;
    constexpr int VEC = E::VEC;
    int first = 0x7fffffff, lastm = -1;
    double run0 = prefix;
#pragma unroll
    for (int g = 0; g < kRegionRows; ++g) {
        float tv[VEC], dv[VEC], m[VEC];
        E::unpack(rt[g], tv);
        E::unpack(rd[g], dv);
        double loc = 0.0;
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            m[e] = fmaxf(-grad_elem(tv[e], dv[e], c, rc), 0.f);
            loc += (double)m[e];
        }
        const double incl = warp_inclusive_scan(loc);
        double run = run0 + (incl - loc);
        const int v0 = v_first + (g * 32 + lane) * VEC;
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            run += (double)m[e];
            if (m[e] > 0.f) {
                lastm = v0 + e;
                if (run > t) first = min(first, v0 + e);
            }
        }
        run0 += __shfl_sync(0xffffffffu, incl, 31);
    }
    first = __reduce_min_sync(0xffffffffu, first);
    lastm = __reduce_max_sync(0xffffffffu, lastm);
    return last || first == 0x7fffffff ? lastm : first;
}

// What the kernel is for.  Errors: first pass only -- row constants, losses and rejection tests; then Draw: the second
// pass over the one row of every sequence that the error-position feedback wants, a cluster to a sequence (of another
// shape than the first pass had, so that a total may round otherwise in fp64).  Hint: the second pass also sums the
// squared distance to the hint.  Ensemble: the units are those of the ensemble feedback (see UnitRef); nothing is
// verified or drawn.
enum HeldMode { kHeldStep = 0, kHeldErrors = 1, kHeldHint = 2, kHeldEnsemble = 3, kHeldDraw = 4, kHeldModes = 5 };

// cand: workspace [B*(k+1)] (step and hint).
template <int DT, int N, int MODE>
__global__ void __launch_bounds__(kHeldThreads, 1)
sd_held_kernel(const __grid_constant__ Params P, HeldCandidate* const cand) {
    using E = Elem<DT>;
    using ET = typename E::type;
    constexpr int VEC = E::VEC;
    constexpr bool STATS = MODE == kHeldErrors, HINT = MODE == kHeldHint, ENS = MODE == kHeldEnsemble, DRAW = MODE == kHeldDraw;
    __shared__ HeldShared sh;
    await_previous_kernel();
    launch_dependents();
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cluster_arrive();                                      // (waited for before the first remote store)

    int unit = (int)blockIdx.x / C;
    bool ok = true;                                        // (range checks; all threads go on to the cluster's barriers)
    if constexpr (DRAW) {
        // of the sequence, the first rejected row (the bonus row if there is none)
        const int b = unit;
        ok = SD_IN(b, P.B, 22);
        unit = b * (P.k + 1) + P.k;
        for (int i0 = 0; ok && i0 < P.k; i0 += 32) {
            const unsigned m = __ballot_sync(0xffffffffu, i0 + lane < P.k && P.accept[b * P.k + i0 + lane] == 0);
            if (m) { unit = b * (P.k + 1) + i0 + __ffs(m) - 1; break; }
        }
    }
    ok = ok && SD_IN(unit, total_units<ENS>(P), 20);
    const UnitRef ur = unit_ref<ENS>(P, unit);
    const int slots = C * kHeldWarps, slot = rank * kHeldWarps + warp;
    // this warp's regions [r0, r0 + n)
    const int NV = P.V / VEC, NR = P.NR, base = NR / slots, rem = NR - base * slots;
    const int r0 = slot * base + min(slot, rem);
    int n = base + (slot < rem ? 1 : 0);
    // (without regions a warp neither loads nor stores: what is read of a row is where its gradient and its hint lie, too)
    if (!ok || !SD_IN(ur.t_row, (long long)P.B * (P.k + 1), 10) || !SD_IN(ur.d_row, (long long)P.B * P.k, 11)) n = 0;
    if (n > 0 && !SD_IN((long long)min(NV, (r0 + n) * kRegionVecs) * VEC - 1, P.V, 12)) n = 0;
    const size_t offD = ur.d_row * P.V;
    const uint4* const gT = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + ur.t_row * P.V);
    const uint4* const gD = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(ENS ? P.Dn[ur.n] : P.D) + offD);

    // (asked for before anything else: wanted at the end of the chain)
    float uk = 0.f;
    if (!STATS && !ENS && ok) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(uk) : "l"(P.u + (size_t)ur.b * (P.k + 1) + P.k));
    uint4 rt[N][kRegionRows], rd[N][kRegionRows];
    const uint64_t policy = STATS || ENS ? policy_normal() : policy_discard();     // (somebody else reads them too)
#pragma unroll
    for (int j = 0; j < N; ++j) {
#pragma unroll
        for (int g = 0; g < kRegionRows; ++g) {
            const int vi = (r0 + j) * kRegionVecs + g * 32 + lane;
            const bool in = j < n && vi < NV;
            rt[j][g] = E::masked();
            // (a bonus row goes the same way with draft logits of 0, whose sums nobody looks at, and kD = 0)
            rd[j][g] = ur.bonus ? make_uint4(0u, 0u, 0u, 0u) : E::masked();
            held_load(rt[j][g], gT + vi, in, policy);
            held_load(rd[j][g], gD + vi, in && !ur.bonus, policy);
        }
    }
    const bool reports = !DRAW && rank == 0 && warp == 0;
    RowConst rc;
    int32_t first = -1;
    uint32_t word = 0;
    if constexpr (DRAW) {
        if (ok) {
            rc = P.rowc[unit];
            if (lane < P.k) first = P.x[ur.b * P.k + lane];
            word = P.wstatus[ur.b];
        }
    }
    AcceptOperands aop;
    aop.valid = false;
    if (!ENS && ok && reports && lane == 0 && !ur.bonus) aop = load_accept_operands<DT>(P, ur.b, ur.i);

    // ---- first pass: references from the maxima of all the warp holds
    if constexpr (!DRAW) {
        LaneSums ls;
        ls.init();
        float RT = kEmptyRef, RD = kEmptyRef;
        {
            float mT = -INFINITY, mD = -INFINITY;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                mT = fmaxf(mT, region_max<DT>(rt[j]));
                mD = fmaxf(mD, region_max<DT>(rd[j]));
            }
            RT = warp_max_ref(ref_of(mT, P.c));
            RD = warp_max_ref(ref_of(mD, P.c));
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
            if (j < n) {
                float sT, sD, sW;
                const int nv = NV - (r0 + j) * kRegionVecs;
                held_sums<DT, false>(rt[j], rd[j], nv, lane, P.c, RT, RD, sT, sD, sW);
                // masked target entries make a NaN: with the test for them
                if (__any_sync(0xffffffffu, sW != sW)) held_sums<DT, true>(rt[j], rd[j], nv, lane, P.c, RT, RD, sT, sD, sW);
                ls.sT += sT;
                ls.sD += sD;
                ls.w += sW;
            }
        }
        {
            // the warp's partial to every block of the cluster
            const double v = warp_fold_lanes(ls, lane);
            PartialStats mine;
            mine.RT = RT; mine.RD = RD;
            mine.sT = __shfl_sync(0xffffffffu, v, 0);
            mine.sD = __shfl_sync(0xffffffffu, v, 8);
            mine.w = __shfl_sync(0xffffffffu, v, 16);
            cluster_wait();
            if (lane < C) *cluster.map_shared_rank(&sh.part[slot], lane) = mine;
            __syncwarp();
        }
        cluster_arrive();
        cluster_wait();
        if (warp == 0) {
            const PartialStats row = held_merge(sh.part, slots, lane);
            if (lane == 0) { sh.row = row; sh.rc = row_constants(P, ur.bonus, row); }
        }
        __syncthreads();
        rc = sh.rc;
    } else {
        cluster_wait();
    }
    if constexpr (STATS) {
        // (the status words are written by the kernel of the drawn rows)
        if (reports && lane == 0) finish_row(P, ur.b, ur.i, sh.row, rc, aop, row_logs(sh.row));
        return;
    } else {
        // ---- second pass, and a third one, of p_n's masses, if max(0, p - q) has none
        void* const gbase = ENS ? P.Gn[ur.n] : P.grad;
        ET* gdst = (gbase && !ur.bonus) ? reinterpret_cast<ET*>(gbase) + (DRAW ? (size_t)ur.b * P.V : offD) : nullptr;
        if (DRAW && gbase && ur.bonus) {
            // no error position: a zero row
            uint4* const z = reinterpret_cast<uint4*>(reinterpret_cast<ET*>(gbase) + (size_t)ur.b * P.V);
            for (int vi = r0 * kRegionVecs + lane; vi < min(NV, (r0 + n) * kRegionVecs); vi += 32) __stcs(z + vi, make_uint4(0u, 0u, 0u, 0u));
        }
        const uint4* const gH = HINT ? reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.hint) + offD) : nullptr;
        if constexpr (ENS) {
            if (reports && lane == 0) finish_row_ensemble(P, ur, sh.row);
            if (!gdst) return;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (j < n) {
                    const int v0 = (r0 + j) * kRegionVecs;
                    float unused = 0.f;
                    pass2_region_impl<DT, false, false, false>(rt[j], rd[j], min(kRegionVecs, NV - v0), lane, P.c, rc, gdst + (size_t)v0 * VEC,
                                                               rt[j], unused);
                }
            }
            return;
        }
        uint32_t flags = 0;
        bool last_ticket = false;
        for (int round = 0;; ++round) {
            float m[N], herr = 0.f;
            double total = 0.0;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                m[j] = 0.f;
                if (j < n) {
                    const int v0 = (r0 + j) * kRegionVecs, nv = min(kRegionVecs, NV - v0);
                    uint4 hq[kRegionRows];
                    if constexpr (HINT) {
#pragma unroll
                        for (int g = 0; g < kRegionRows; ++g)
                            hq[g] = (!ur.bonus && round == 0 && g * 32 + lane < nv) ? __ldcs(gH + v0 + g * 32 + lane) : make_uint4(0u, 0u, 0u, 0u);
                    }
                    m[j] = pass2_region_impl<DT, false, HINT>(rt[j], rd[j], nv, lane, P.c, rc, gdst ? gdst + (size_t)v0 * VEC : nullptr,
                                                              HINT ? hq : rt[j], herr);
                    total += (double)m[j];
                }
            }
            if constexpr (HINT) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) herr += __shfl_xor_sync(0xffffffffu, herr, off);
            }
            double2* const mass = sh.mass[round];
            if (lane < C) *cluster.map_shared_rank(&mass[slot], lane) = make_double2(total, (double)herr);
            __syncwarp();
            cluster_arrive();
            if (reports && round == 0 && lane == 0) finish_row(P, ur.b, ur.i, sh.row, rc, aop, row_logs(sh.row));
            __syncwarp();
            cluster_wait();

            // every warp finds the owner of u * total on its own, all from the same sums in the same order
            const int per = (slots + 31) / 32;
            const int s0 = min(slots, lane * per), s1 = min(slots, s0 + per);
            double held = 0.0;
            for (int s = s0; s < s1; ++s) held += mass[s].x;
            const double incl = warp_inclusive_scan(held);
            const double all = __shfl_sync(0xffffffffu, incl, 31);
            if (rank == 0 && warp == 1 && round == 0 && !ur.bonus && SD_IN(ur.d_row, (long long)P.B * P.k, 21)) {
                if (P.acc_prob && lane == 0) P.acc_prob[ur.d_row] = (float)(1.0 - all * (double)P.tau);
                if constexpr (HINT) {
                    double e = 0.0;
                    for (int s = s0; s < s1; ++s) e += mass[s].y;
                    e = warp_sum(e);
                    if (lane == 0) P.hint_err[ur.d_row] = (float)e;
                }
            }
            int y = 0;
            bool mine;
            if (!(all > 0.0) || !isfinite(all)) {
                if (round == 0 && !ur.bonus) {             // (the same for every warp of the cluster)
                    flags |= SD_STATUS_ZERO_RESIDUAL;
                    rc.kD = rc.negRD = 0.f;                // (as on a bonus row)
#pragma unroll
                    for (int j = 0; j < N; ++j)
#pragma unroll
                        for (int g = 0; g < kRegionRows; ++g) rd[j][g] = make_uint4(0u, 0u, 0u, 0u);
                    gdst = nullptr;
                    continue;
                }
                if (ur.bonus) flags |= SD_STATUS_BAD_ROW;
                mine = slot == 0;
            } else {
                const double t = (double)uk * all;
                int owner = 0x7fffffff, last = -1;
                double run = incl - held, prefix = 0.0;
                for (int s = s0; s < s1; ++s) {
                    const double x = mass[s].x, next = run + x;
                    if (x > 0.0) last = s;
                    if (owner == 0x7fffffff && next > t) { owner = s; prefix = run; }
                    run = next;
                }
                const unsigned has = __ballot_sync(0xffffffffu, owner != 0x7fffffff);
                const bool past_end = has == 0;            // rounding pushed u * total to the total: the last entry with mass
                const int src = has ? __ffs(has) - 1 : 0;
                owner = __shfl_sync(0xffffffffu, owner, src);
                prefix = __shfl_sync(0xffffffffu, prefix, src);
                if (past_end) owner = __reduce_max_sync(0xffffffffu, last);
                mine = owner == slot;
                if (mine) {
                    // the region, then the entry
                    int at = -1, lastj = -1;
                    double before = prefix;
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        if (m[j] > 0.f) lastj = j;
                        if (at < 0) {
                            const double next = before + (double)m[j];
                            if (next > t) at = j;
                            else before = next;
                        }
                    }
                    const bool to_last = past_end || at < 0;
                    if (to_last) at = lastj;
                    uint4 ft[kRegionRows], fd[kRegionRows];
#pragma unroll
                    for (int g = 0; g < kRegionRows; ++g) { ft[g] = rt[0][g]; fd[g] = rd[0][g]; }
#pragma unroll
                    for (int j = 1; j < N; ++j)
                        if (at == j) {
#pragma unroll
                            for (int g = 0; g < kRegionRows; ++g) { ft[g] = rt[j][g]; fd[g] = rd[j][g]; }
                        }
                    y = held_search<DT>(ft, fd, (r0 + max(at, 0)) * kRegionVecs * VEC, lane, P.c, rc, before, t, to_last);
                    if (y < 0) y = 0;
                }
            }
            if constexpr (DRAW) {
                if (mine && ok) held_emit(P, ur.b, ur.i, y, word | flags, first, lane);
                return;
            }
            // two tickets of a unit: its row report, its candidate
            uint32_t tickets = reports ? 1u : 0u;
            if (mine) {
                ++tickets;
                if (lane == 0 && ok)
                    *reinterpret_cast<int2*>(cand + unit) = make_int2(y, (int)flags);
            }
            if (tickets && ok) {
                int got = 0;
                if (lane == 0) got = take_tickets(P, ur.b, tickets) ? 1 : 0;
                last_ticket = __shfl_sync(0xffffffffu, got, 0) != 0;
                __syncwarp();
            }
            break;
        }
        if (last_ticket) held_finish(P, cand, ur.b, lane);
    }
}

}  // namespace sdv
