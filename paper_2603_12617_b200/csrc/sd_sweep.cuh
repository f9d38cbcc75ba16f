// The step as two sweeps over the logits, grids of small independent blocks: no cluster, no ring, nobody
// waits for anybody.  A unit (sequence, row) is cut into `slices` items of the same number of sampling
// regions (towards the end of a sweep smaller ones), a block takes one item, a warp every eighth region of it, straight from global memory into
// registers.  Three kernels, each of which comes in as the one before goes out:
//
//   sd_sweep_stats_kernel  softmax sums of every item to the workspace.
//   sd_sweep_rows_kernel   merges the items of every row in slice order and reports the rows: constants,
//                          losses, rejection tests.
//   sd_sweep_grad_kernel   gradient of every pair row; masses of the sampling regions only for the one row
//                          per sequence that the extra token is drawn from (bonus rows that are not drawn
//                          from cost nothing).  The block that brings that row's last item draws.
//
// The second sweep runs through the items backwards: what the first one read last, and asked L2 to keep,
// is still there.
//
// What bounds it: HBM, the exponentials close behind.  Measured alone, the first sweep's loop reads 5.6 TB/s
// and the second's reads and writes 6.1 TB/s; their arithmetic (144 and 141 instructions per region and
// warp, 64 cycles of exponentials per region and SM) hides behind the copies with 48 warps an SM.
// sd_stream_kernel reads every logit from HBM once, but its 28 consumer warps share one ring and all blocks
// read at the same time and compute at the same time, so at bf16, where the exponentials take as long as
// the reads, it moves 2.9 TB/s.  Step on 32 sequences, 8 draft tokens, 128 256 bf16 entries: 71.1 us there,
// 55.6 us here; 64 sequences, 4 tokens, 151 936: 93.4 and 69.0 us; 8, 5, 128 256: 35.0 and 18.6.  Of the 57.4 us that the first
// of these took with items of one size, clock stamps of every block: first sweep 29.5, the last 8 with fewer and fewer
// blocks; 4.5 until the second sweep works, 2 of them in the rows kernel; second sweep 24.  16 sequences, 5 tokens, 65 536 bf16
// entries, when it took 19.6 us (18.2 now): 8, 4, 5, and 4 for the draws.
// The rule which of the two a call takes is use_sweeps (host).
//
// Tried and dropped, on the first of these: one persistent kernel whose warps take both passes of an item
// from per-warp rings of bulk copies (82 us: many 1 KiB copies in flight slow each other down) or of
// cp.async (99: their instructions), from registers in teams of blocks that wait for their row (71), and
// from a queue that mixes first and second passes so that the second hits L2 (70; again, on the present loops, with
// sequences opened for the second pass by a flag: 118.  Under load a round trip is 2 to 3 us, and partial, counter, row and
// flag are ten of them: more logits lie between the passes than L2 keeps).  The first sweep of a group of sequences in one
// grid with the second of the group before, a rows kernel between: 60.6 with one group, 68 with two, 80 with three.  L2
// prefetches of a block's or a warp's next regions: 59 to 68.  Items in row order: 57.5.
#pragma once

#include "sd_kernels.cuh"

namespace sdv {

constexpr int kSweepWarps = 8;
constexpr int kSweepThreads = kSweepWarps * 32;
constexpr int kMaxSlices = 32;                  // items of a row: one warp merges them, one per lane
constexpr int kSweepStep = kSweepWarps * kRegionVecs;   // vectors from a warp's region to its next

struct Sweep {
    int slices;              // items per unit (1..kMaxSlices)
    int regions;             // sampling regions per item (the last item of a unit may have fewer)
    int fine_units;          // units from the last one backwards whose items are smaller in the first sweep,
    int fine_rows;           // pair rows from the first one on whose items are smaller in the second:
    int fine_slices, fine_regions;   // so many of so many regions (slices and regions where there are none)
    int part_stride;         // room for a unit's partials
    PartialStats* part;      // workspace [units][part_stride]; its memory is region_sums' from the second sweep on
    uint32_t* arrived;       // workspace [units], zero on entry and zero again on exit
    int draw_threads;        // of a block that draws
    unsigned kept;           // items, from the last one backwards, that L2 is asked to keep between the sweeps
    int all_rows;            // second sweep: masses of every row wanted (acceptance probabilities)
    int draw_blocks;         // second sweep: its first blocks, those of the rows that are drawn from,
    int draw_slices;         // ... the items of such a row
    int draw_regions;        // ... and their sampling regions
};

// What the second sweep is for.
enum SweepMode { kSweepStepMode = 0, kSweepErrors = 1, kSweepHint = 2 };

__device__ __forceinline__ uint4 load_l2(const uint4* p, uint64_t policy) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy));
    return v;
}
// The same for vectors that the neighbouring lane reads too (kept in L1).
__device__ __forceinline__ uint4 load_l2_shared(const uint4* p, uint64_t policy) {
    uint4 v;
    asm volatile("ld.global.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy));
    return v;
}

// Sums of the lanes of a warp that share the references (RT, RD) into *out, in fp64 and a fixed order.
__device__ __forceinline__ void warp_post_lanes(const LaneSums& ls, float RT, float RD, int lane, PartialStats* out) {
    const double v = warp_fold_lanes(ls, lane);
    if (lane == 0) { out->RT = RT; out->RD = RD; out->sT = v; }
    if (lane == 8) out->sD = v;
    if (lane == 16) out->w = v;
}

// raise_references for every region of a row: maxima and a vote, the rest only where an entry is above the
// references (the same references and sums).
template <int DT, bool BONUS>
__device__ __forceinline__ void follow_references(const uint4 (&rt)[kRegionRows], const uint4 (&rd)[kRegionRows], float c, Pass1State& s) {
    const float t = region_max<DT>(rt), d = BONUS ? 0.f : region_max<DT>(rd);
    if (!__any_sync(0xffffffffu, __fmul_rn(t, c) > s.RT || (!BONUS && __fmul_rn(d, c) > s.RD))) return;
    const float nT = fmaxf(s.RT, warp_max_ref(ref_of(t, c)));
    const float nD = BONUS ? kEmptyRef : fmaxf(s.RD, warp_max_ref(ref_of(d, c)));
    s.ls.rescale(nT - s.RT, nD - s.RD);
    s.RT = nT;
    s.RD = nD;
}

__device__ __forceinline__ PartialStats load_partial_cg(const PartialStats* p) {
    PartialStats r;
    const float4 a = __ldcg(reinterpret_cast<const float4*>(p)), b = __ldcg(reinterpret_cast<const float4*>(p) + 1);
    memcpy(&r, &a, 16);
    memcpy(reinterpret_cast<char*>(&r) + 16, &b, 16);
    return r;
}

// ---- rows that are not whole 16-byte vectors --------------------------------------------------
// Such a row starts anywhere within a vector, and a target row elsewhere than its draft row.  The regions
// of a row pair are laid out on the vectors of the draft row (and the gradient, which starts at the same
// place), the target's entries are moved into place: two neighbouring vectors and a funnel shift that is
// the same for the whole row, 15 instructions for 8 bf16 pairs.  A bonus row is laid out on itself.
// Regions at the ends of a row, where a vector would reach into another row or out of the tensor, are read
// and written entry by entry, out of line and with registers of their own: with one set for both, filled by a
// function for the ends, every region went through local memory (13 sequences, 8 tokens, 110 593 fp32 entries 67.3 us,
// 40 since; 122, 4, 119 177 302 and 200; 64, 4, 100 001 bf16 84.9 and 60).  16 sequences, 5 tokens, 50 257 bf16
// entries: 19.3 us, against 91.6 us for the element-wise kernel, whose one block per row reads two bytes a lane.
template <int DT> struct RowFrame {
    const typename Elem<DT>::type *rowT, *rowD;
    const uint4 *T16, *D16;      // vector 0 of the regions, aligned: up to a vector before the row
    int lead;                    // entries of vector 0 before the row
    int shift;                   // entries the target's vectors start before the draft's
    int nvec;                    // vectors of the row
};
template <int DT>
__device__ __forceinline__ int entry_phase(const void* p) {
    return (int)((reinterpret_cast<uintptr_t>(p) / sizeof(typename Elem<DT>::type)) & (Elem<DT>::VEC - 1));
}
template <int DT>
__device__ __forceinline__ RowFrame<DT> row_frame(const Params& P, const UnitRef& ur) {
    constexpr int VEC = Elem<DT>::VEC;
    using ET = typename Elem<DT>::type;
    RowFrame<DT> f;
    f.rowT = reinterpret_cast<const ET*>(P.T) + ur.t_row * P.V;
    f.rowD = reinterpret_cast<const ET*>(P.D) + ur.d_row * P.V;
    const int pt = entry_phase<DT>(f.rowT);
    f.lead = ur.bonus ? pt : entry_phase<DT>(f.rowD);
    f.shift = (pt - f.lead) & (VEC - 1);
    f.T16 = reinterpret_cast<const uint4*>(f.rowT - f.lead - f.shift);
    f.D16 = reinterpret_cast<const uint4*>(f.rowD - f.lead);
    f.nvec = (P.V + f.lead + VEC - 1) / VEC;
    return f;
}
// Does the region that starts at vector v lie in the row with every vector that is read for it?
template <int DT>
__device__ __forceinline__ bool inner_region(const RowFrame<DT>& f, int V, int v) {
    return v > 0 && (v + kRegionVecs + (f.shift ? 1 : 0)) * Elem<DT>::VEC - f.lead - f.shift <= V;
}
template <int DT>
__device__ __forceinline__ uint4 funnel(const uint4& a, const uint4& b, int shift) {
    const int bytes = shift * (int)sizeof(typename Elem<DT>::type);
    uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = (bytes & 8) ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = (bytes & 4) ? w[i + 1] : w[i];
    if constexpr (DT == SD_DTYPE_F32) return make_uint4(w[0], w[1], w[2], w[3]);
    const int bits = (bytes & 2) * 8;
    return make_uint4(__funnelshift_r(w[0], w[1], bits), __funnelshift_r(w[1], w[2], bits), __funnelshift_r(w[2], w[3], bits),
                      __funnelshift_r(w[3], w[4], bits));
}
// (checked build) Every entry of the vectors that load_inner reads is one of its row.
template <int DT, bool BONUS>
__device__ __forceinline__ bool inner_in_bounds(const RowFrame<DT>& f, int V, int v) {
    [[maybe_unused]] constexpr int VEC = Elem<DT>::VEC;
    return SD_IN(v * VEC - f.lead - f.shift, V, 16) &&
           SD_IN((v + kRegionVecs + (!BONUS && f.shift ? 1 : 0)) * VEC - f.lead - f.shift - 1, V, 16) &&
           (BONUS || (SD_IN(v * VEC - f.lead, V, 16) && SD_IN((v + kRegionVecs) * VEC - f.lead - 1, V, 16)));
}
// An inner region.
template <int DT, bool BONUS>
__device__ __forceinline__ void load_inner(const RowFrame<DT>& f, int v, int lane, uint64_t policy, uint4 (&rt)[kRegionRows],
                                           uint4 (&rd)[kRegionRows]) {
    uint4 next[kRegionRows];
    const bool shifted = !BONUS && f.shift;
#pragma unroll
    for (int g = 0; g < kRegionRows; ++g) {
        rt[g] = load_l2_shared(f.T16 + v + g * 32 + lane, policy);
        if (!BONUS) rd[g] = load_l2(f.D16 + v + g * 32 + lane, policy);
        if (shifted) next[g] = load_l2_shared(f.T16 + v + g * 32 + lane + 1, policy);
    }
    if (shifted) {
#pragma unroll
        for (int g = 0; g < kRegionRows; ++g) rt[g] = funnel<DT>(rt[g], next[g], f.shift);
    }
}
// Any region, entry by entry; what is not in the row reads as -inf.
template <int DT, bool BONUS>
__device__ __forceinline__ void load_edge(const RowFrame<DT>& f, int V, int v, int lane, uint4 (&rt)[kRegionRows], uint4 (&rd)[kRegionRows]) {
    using E = Elem<DT>;
    constexpr int VEC = E::VEC;
#pragma unroll
    for (int g = 0; g < kRegionRows; ++g) {
        float t[VEC], d[VEC];
        const int e0 = (v + g * 32 + lane) * VEC - f.lead;
#pragma unroll
        for (int z = 0; z < VEC; ++z) {
            const bool in = e0 + z >= 0 && e0 + z < V;
            t[z] = in && SD_IN(e0 + z, V, 17) ? E::load(f.rowT, e0 + z) : -INFINITY;
            d[z] = (!BONUS && in) ? E::load(f.rowD, e0 + z) : -INFINITY;
        }
        rt[g] = E::pack(t);              // (bf16 values come back as they were)
        rd[g] = E::pack(d);
    }
}
// Both passes over a region at an end of the row, out of line: all of its vectors' registers are these functions' own,
// and the loops over inner regions keep to theirs.
template <int DT, bool BONUS>
__device__ __noinline__ Pass1State edge_pass1(const RowFrame<DT> f, int V, int v, int lane, float c, Pass1State s) {
    uint4 rt[kRegionRows], rd[kRegionRows];
    load_edge<DT, BONUS>(f, V, v, lane, rt, rd);
    follow_references<DT, BONUS>(rt, rd, c, s);
    float sT, sD, sW;
    region_sums_of<DT, BONUS, true>(rt, rd, c, s.RT, s.RD, sT, sD, sW);
    s.ls.sT += sT;
    s.ls.sD += sD;
    s.ls.w += sW;
    return s;
}
template <int DT, bool BONUS, bool MASS>
__device__ __noinline__ float edge_pass2(const RowFrame<DT> f, int V, int v, typename Elem<DT>::type* grow, int lane, float c, const RowConst rc) {
    using E = Elem<DT>;
    constexpr int VEC = E::VEC;
    uint4 rt[kRegionRows], rd[kRegionRows];
    float unused = 0.f;
    load_edge<DT, BONUS>(f, V, v, lane, rt, rd);
    const float mass = pass2_region_impl<DT, BONUS, false, MASS>(rt, rd, kRegionVecs, lane, c, rc, nullptr, rt, unused);
    if (!BONUS && grow) {
#pragma unroll
        for (int g = 0; g < kRegionRows; ++g) {
            float t[VEC], d[VEC];
            E::unpack(rt[g], t);
            E::unpack(rd[g], d);
            const int e0 = (v + g * 32 + lane) * VEC - f.lead;
#pragma unroll
            for (int z = 0; z < VEC; ++z)
                if (e0 + z >= 0 && e0 + z < V && SD_IN(e0 + z, V, 18)) E::store(grow, e0 + z, grad_elem(t[z], d[z], c, rc));
        }
    }
    return mass;
}

template <int DT, bool BONUS>
__device__ __forceinline__ void ragged_pass1(const RowFrame<DT>& f, int V, int v0, int v1, int lane, float c, uint64_t policy,
                                             Pass1State& s) {
    for (int v = v0; v < v1; v += kSweepStep) {
        if (!inner_region<DT>(f, V, v)) {
            s = edge_pass1<DT, BONUS>(f, V, v, lane, c, s);
            continue;
        }
        uint4 rt[kRegionRows], rd[kRegionRows];
        if (!inner_in_bounds<DT, BONUS>(f, V, v)) continue;
        load_inner<DT, BONUS>(f, v, lane, policy, rt, rd);
        follow_references<DT, BONUS>(rt, rd, c, s);     // (every region, as the element-wise kernel does)
        float sT = 0.f, sD = 0.f, sW = 0.f;
        region_sums_of<DT, BONUS, false>(rt, rd, c, s.RT, s.RD, sT, sD, sW);
        // masked target entries (a NaN): with the test for them
        if (__any_sync(0xffffffffu, sW != sW)) region_sums_of<DT, BONUS, true>(rt, rd, c, s.RT, s.RD, sT, sD, sW);
        s.ls.sT += sT;
        s.ls.sD += sD;
        s.ls.w += sW;
    }
}

// Pass 2; grow = the gradient row, or null.  v1 may lie past the row: regions that this row does not have, but
// rows that start later within a vector do, get the mass 0.
template <int DT, bool BONUS, bool MASS>
__device__ __forceinline__ void ragged_pass2(const RowFrame<DT>& f, int V, int v0, int v1, typename Elem<DT>::type* grow, float* rsum,
                                             int lane, float c, const RowConst& rc) {
    constexpr int VEC = Elem<DT>::VEC;
    for (int v = v0; v < v1; v += kSweepStep) {
        float mass = 0.f, unused = 0.f;
        if (v >= f.nvec) {
            if (!MASS) break;
        } else if (inner_region<DT>(f, V, v)) {
            uint4 rt[kRegionRows], rd[kRegionRows];
            if (!inner_in_bounds<DT, BONUS>(f, V, v)) continue;       // (the gradient lies where the draft does)
            load_inner<DT, BONUS>(f, v, lane, policy_discard(), rt, rd);
            mass = pass2_region_impl<DT, BONUS, false, MASS>(rt, rd, kRegionVecs, lane, c, rc,
                                                             grow ? grow + (size_t)v * VEC - f.lead : nullptr, rt, unused);
        } else {
            mass = edge_pass2<DT, BONUS, MASS>(f, V, v, grow, lane, c, rc);
        }
        if constexpr (MASS) {
            if (lane == 0) *rsum = mass;
            rsum += kSweepWarps;
        }
    }
}

// Pass 1 of a warp's regions of an item: gT and gD lead to the first of them, `nvec` vectors of the item lie
// from there on, the next region `step` vectors further.  (Fetching the next region while this one is worked on was
// measured as well: no faster, the other warps of the SM hide the loads.)
// The references come from the warp's first region, which costs least, but an entry far above them has an
// exponent as large, rounded as coarsely.  RAISE: every region raises them, so that no exponent is above 0,
// for callers with few warps, hence few references, to a row.
template <int DT, bool BONUS, bool RAISE = false>
__device__ __forceinline__ void sweep_pass1(const uint4* gT, const uint4* gD, int nvec, int step, int lane, float c, uint64_t policy,
                                            Pass1State& s) {
    constexpr float kTooLarge = 1.152921504606846976e18f;   // 2^60
    bool first = true;
    for (; nvec >= kRegionVecs; gT += step, gD += step, nvec -= step, first = false) {
        uint4 rt[kRegionRows], rd[kRegionRows];
#pragma unroll
        for (int g = 0; g < kRegionRows; ++g) {
            rt[g] = load_l2(gT + g * 32 + lane, policy);
            if (!BONUS) rd[g] = load_l2(gD + g * 32 + lane, policy);
        }
        if (RAISE)      follow_references<DT, BONUS>(rt, rd, c, s);
        else if (first) raise_references<DT, BONUS>(rt, rd, c, s);
        float sT, sD, sW;
        region_sums_of<DT, BONUS, false>(rt, rd, c, s.RT, s.RD, sT, sD, sW);
        // masked target entries (NaN) or entries far above the references: maxima first, then the sums
        if (__any_sync(0xffffffffu, (!RAISE && (!(sT < kTooLarge) || !(sD < kTooLarge))) || sW != sW)) {
            s = pass1_region_again<DT, BONUS>(gT, gD, kRegionVecs, lane, c, s);
            continue;
        }
        s.ls.sT += sT;
        s.ls.sD += sD;
        s.ls.w += sW;
    }
    if (nvec > 0) s = pass1_region_again<DT, BONUS>(gT, gD, nvec, lane, c, s);   // cut short by the end of the row
}

// The same with two regions of a warp on their way at a time, and every region raising the references: for warps with few
// regions, whose time is round trips.
template <int DT, bool BONUS>
__device__ __forceinline__ void sweep_pass1_pairs(const uint4* gT, const uint4* gD, int nvec, int step, int lane, float c, uint64_t policy,
                                                  Pass1State& s) {
    for (; nvec >= kRegionVecs; gT += 2 * step, gD += 2 * step, nvec -= 2 * step) {
        uint4 rt[2][kRegionRows], rd[2][kRegionRows];
        const bool both = nvec - step >= kRegionVecs;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int g = 0; g < kRegionRows; ++g) {
                rt[j][g] = rd[j][g] = Elem<DT>::masked();
                if (j == 0 || both) {
                    rt[j][g] = load_l2(gT + j * step + g * 32 + lane, policy);
                    if (!BONUS) rd[j][g] = load_l2(gD + j * step + g * 32 + lane, policy);
                }
            }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (j == 1 && !both) break;
            follow_references<DT, BONUS>(rt[j], rd[j], c, s);
            float sT, sD, sW;
            region_sums_of<DT, BONUS, false>(rt[j], rd[j], c, s.RT, s.RD, sT, sD, sW);
            // masked target entries (a NaN): with the test for them
            if (__any_sync(0xffffffffu, sW != sW)) region_sums_of<DT, BONUS, true>(rt[j], rd[j], c, s.RT, s.RD, sT, sD, sW);
            s.ls.sT += sT;
            s.ls.sD += sD;
            s.ls.w += sW;
        }
        if (!both && nvec > step) { gT += step; gD += step; nvec -= step; break; }
    }
    if (nvec > 0) s = pass1_region_again<DT, BONUS>(gT, gD, nvec, lane, c, s);   // cut short by the end of the row
}

// One block per item: blockIdx.x = unit, blockIdx.y = slice.  FINE (a grid of one dimension): the units with large items like
// that, then those with small ones.
template <int DT, bool RAGGED, bool FINE>
__global__ void __launch_bounds__(kSweepThreads, !RAGGED ? 6 : DT == SD_DTYPE_F32 ? 6 : 5)
sd_sweep_stats_kernel(const __grid_constant__ Params P, const __grid_constant__ Sweep S) {
    using E = Elem<DT>;
    using ET = typename E::type;
    __shared__ PartialStats wpart[kSweepWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    await_previous_kernel();                         // (first: the rows kernel reads inputs before its own wait)
    launch_dependents();
    int unit = blockIdx.x, slice = blockIdx.y, regions = S.regions;
    unsigned behind = (gridDim.y - 1u - blockIdx.y) * gridDim.x + (gridDim.x - 1u - blockIdx.x);     // items
    if constexpr (FINE) {
        int units = total_units<false>(P) - S.fine_units;
        const int large = units * S.slices;
        if (unit < large) {
            slice = unit / units;
            unit -= slice * units;
            behind -= S.fine_units * S.fine_slices / 2;           // (of about half as many regions each)
        } else {
            slice = (unit - large) / S.fine_units;
            unit = unit - large - slice * S.fine_units + units;
            regions = S.fine_regions;
            behind /= 2;
        }
    }
    const uint64_t policy = behind < S.kept ? policy_keep() : policy_discard();
    const int at = unit * S.part_stride + slice;
    const UnitRef ur = unit_ref<false>(P, unit);
    const int v0 = (slice * regions + warp) * kRegionVecs;
    Pass1State ps;
    ps.RT = ps.RD = kEmptyRef;
    ps.ls.init();
    if constexpr (RAGGED) {
        const RowFrame<DT> f = row_frame<DT>(P, ur);
        int v1 = min((slice + 1) * regions * kRegionVecs, f.nvec);
        if (!SD_IN(ur.t_row, (long long)P.B * (P.k + 1), 10) || !SD_IN(ur.d_row, (long long)P.B * P.k, 11)) v1 = 0;
        if (ur.bonus) ragged_pass1<DT, true>(f, P.V, v0, v1, lane, P.c, policy, ps);
        else          ragged_pass1<DT, false>(f, P.V, v0, v1, lane, P.c, policy, ps);
    } else {
        int nvec = min((slice + 1) * regions * kRegionVecs, P.V / E::VEC) - v0;
        if (nvec > 0 && !SD_IN((long long)(v0 + nvec) * E::VEC - 1, P.V, 10)) nvec = 0;
        if (!SD_IN(ur.t_row, (long long)P.B * (P.k + 1), 10) || !SD_IN(ur.d_row, (long long)P.B * P.k, 11)) nvec = 0;
        const uint4* const gT = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + ur.t_row * P.V) + v0;
        const uint4* const gD = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.D) + ur.d_row * P.V) + v0;
        if (ur.bonus) sweep_pass1<DT, true>(gT, gD, nvec, kSweepStep, lane, P.c, policy, ps);
        else          sweep_pass1<DT, false>(gT, gD, nvec, kSweepStep, lane, P.c, policy, ps);
    }
    warp_post_lanes(ps.ls, ps.RT, ps.RD, lane, &wpart[warp]);
    __syncthreads();
    if (warp == 0) {
        const PartialStats item = warp_merge_lanes(lane < kSweepWarps ? wpart[lane] : empty_partial());
        if (lane == 0 && SD_IN(at, (long long)total_units<false>(P) * S.part_stride, 26)) S.part[at] = item;
    }
}

// A block per sequence, a warp per row (up to kRowsMaxWarps of them at a time).  Leaves the sequence's first rejected
// position (k if there is none) in P.accept[b * k].  MANY: held to 40 registers, six blocks of eight warps to an SM (rule and
// figures: launch_sweeps_of, host).
constexpr int kRowsMaxWarps = 16;
template <int DT, bool MANY>
__global__ void __launch_bounds__(kRowsMaxWarps * 32, MANY ? 3 : 0)
sd_sweep_rows_kernel(const __grid_constant__ Params P, const __grid_constant__ Sweep S) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = (int)blockDim.x >> 5;
    const int b = blockIdx.x;
    __shared__ uint8_t accepted[SD_MAX_K];
    launch_dependents();
    for (int i = warp; i <= P.k; i += warps) {
        const int unit = b * (P.k + 1) + i;
        AcceptOperands aop;
        aop.valid = false;
        if (lane == 0 && i < P.k) aop = load_accept_operands<DT>(P, b, i);   // (inputs of the call)
        const int slices = unit < total_units<false>(P) - S.fine_units ? S.slices : S.fine_slices;
        const bool mine = lane < slices && SD_IN(unit, total_units<false>(P), 26);
        const PartialStats* const part = S.part + (size_t)unit * S.part_stride + lane;
        await_previous_kernel();
        const PartialStats row = warp_merge_lanes(mine ? load_partial_cg(part) : empty_partial());
        const RowLogs logs = warp_row_logs(row);
        if (lane == 0) {
            if (P.status && i == 0 && SD_IN(b, P.B, 21)) P.status[b] = 0;      // the words are ORed in by the second sweep
            const bool acc = finish_row(P, b, i, row, row_constants(P, i == P.k, row), aop, logs);
            if (i < P.k) accepted[i] = acc;
        }
    }
    __syncthreads();
    if (warp != 0) return;
    int n = P.k;
    for (int i0 = 0; i0 < P.k; i0 += 32) {
        const unsigned m = __ballot_sync(0xffffffffu, i0 + lane < P.k && !accepted[i0 + lane]);
        if (m) { n = i0 + __ffs(m) - 1; break; }
    }
    if (lane == 0 && SD_IN(b * P.k, P.B * P.k, 22)) P.accept[b * P.k] = (uint8_t)n;
}

// Pass 2 of a warp's regions of an item.
template <int DT, bool BONUS, bool HINT, bool MASS>
__device__ __forceinline__ void sweep_pass2(const uint4* gT, const uint4* gD, const uint4* gH, typename Elem<DT>::type* gdst,
                                            float* rsum, int nvec, int lane, float c, uint64_t policy, const RowConst& rc,
                                            float& herr) {
    using E = Elem<DT>;
    for (; nvec > 0; gT += kSweepStep, gD += kSweepStep, nvec -= kSweepStep) {
        uint4 rt[kRegionRows], rd[kRegionRows], hq[kRegionRows];
        float mass;
        if (nvec >= kRegionVecs) {
#pragma unroll
            for (int g = 0; g < kRegionRows; ++g) {
                rt[g] = load_l2(gT + g * 32 + lane, policy);
                if (!BONUS) rd[g] = load_l2(gD + g * 32 + lane, policy);
                if (HINT) hq[g] = __ldcs(gH + g * 32 + lane);
            }
            mass = pass2_region_impl<DT, BONUS, HINT, MASS>(rt, rd, kRegionVecs, lane, c, rc, gdst, hq, herr);
        } else {
#pragma unroll
            for (int g = 0; g < kRegionRows; ++g) {
                const int vi = g * 32 + lane;
                rt[g] = vi < nvec ? load_l2(gT + vi, policy) : E::masked();
                rd[g] = (!BONUS && vi < nvec) ? load_l2(gD + vi, policy) : E::masked();
                if (HINT) hq[g] = vi < nvec ? __ldcs(gH + vi) : make_uint4(0u, 0u, 0u, 0u);
            }
            mass = pass2_region_impl<DT, BONUS, HINT, MASS>(rt, rd, nvec, lane, c, rc, gdst, hq, herr);
        }
        if constexpr (MASS) {
            if (lane == 0) *rsum = mass;
            rsum += kSweepWarps;
        }
        if (gdst) gdst += (size_t)kSweepStep * E::VEC;
        if (HINT) gH += kSweepStep;
    }
}

// ---- the draw -----------------------------------------------------------------------------------
// A draw is done by a team, the first T threads of a block.
template <int T>
__device__ __forceinline__ void team_sync() {
    if constexpr (T == kSweepThreads) __syncthreads();
    else asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
}

// Sums of the team's threads before a thread's own, and of all of them, in a fixed order.  `sums` is free again after
// the team's next barrier.
template <int T>
__device__ __noinline__ double team_sums_before(double mine, double* sums, double* all) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double incl = warp_inclusive_scan(mine);
    if (lane == 31) sums[warp] = incl;
    team_sync<T>();
    double warps = lane < T / 32 ? sums[lane] : 0.0;
#pragma unroll
    for (int off = 1; off < T / 32; off <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, warps, off);
        if (lane >= off) warps += o;
    }
    *all = __shfl_sync(0xffffffffu, warps, T / 32 - 1);
    const double before = __shfl_sync(0xffffffffu, warps, max(warp - 1, 0));
    return (warp > 0 ? before : 0.0) + (incl - mine);
}

// Where a rejection leaves no residual mass: an entry drawn from p_n, in every thread.  There are no region masses of p_n, so
// every warp adds up a share of the row and the one into whose share the draw falls takes it once more, region by
// region; sums, prefixes and totals in fp64, from the entries on.  Round trips are all it consists of, eight loads each: 40 sequences
// whose draws all come here, rows of 131 072 bf16 entries, 130 us for the call (one warp 548); 16 of 50 257 35 (696).
template <int DT, int T>
__device__ __noinline__ int sweep_draw_from_p(const Params& P, const RowConst& rc, size_t offT, double u, int lead) {
    using E = Elem<DT>;
    constexpr int kEntries = kRegionVecs * E::VEC, PER = kEntries / 32, kWarps = T / 32;
    __shared__ double share[kWarps];
    __shared__ int drawn;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (P.NR + kWarps - 1) / kWarps, j0 = min(P.NR, warp * per), j1 = min(P.NR, j0 + per);
    const auto logit = [&](int v) {                      // (no branch: the loads of eight entries go out together)
        const float z = E::load(P.T, offT + min(max(v, 0), P.V - 1));
        return v >= 0 && v < P.V ? z : -INFINITY;
    };
    // mass of n entries, eight loads at a time, from v on and `step` apart
    const auto lane_sum = [&](int v, int step, int n) {
        double s = 0.0;
        for (int i = 0; i < n; i += 8) {
            float z[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) z[q] = logit(v + (i + q) * step);
#pragma unroll
            for (int q = 0; q < 8; ++q) s += (double)prob_elem(z[q], P.c, rc);
        }
        return s;
    };
    double mine = warp_sum(lane_sum(j0 * kEntries + lane - lead, 32, (j1 - j0) * PER));
    if (threadIdx.x == 0) drawn = 0;
    if (lane == 0) share[warp] = mine;
    team_sync<T>();
    // the first share whose end exceeds t, or (rounding pushed t to the total) the last one with mass
    double total = 0.0, before = 0.0, run = 0.0;
    for (int w = 0; w < kWarps; ++w) total += share[w];
    const double t = u * total;
    int owner = -1;
    bool found = false;
#pragma unroll 1
    for (int w = 0; w < kWarps && !found; ++w) {
        if (share[w] > 0.0) { owner = w; before = run; found = run + share[w] > t; }
        run += share[w];
    }
    if (warp == owner && isfinite(total)) {
        // the region that the sum exceeds t in, or the last with mass; then the entry
        int region = j0;
        double ahead = before;
        for (int j = j0; j < j1; ++j) {
            const double m = warp_sum(lane_sum(j * kEntries + lane - lead, 32, PER));
            if (m > 0.0) { region = j; ahead = before; }
            before += m;
            if (before > t) break;
        }
        const int v0 = region * kEntries + lane * PER - lead;
        double sum = lane_sum(v0, 1, PER);
        sum = ahead + (warp_inclusive_scan(sum) - sum);
        int first = 0x7fffffff, last = -1;
#pragma unroll 1
        for (int e = 0; e < PER; ++e) {
            const double m = (double)prob_elem(logit(v0 + e), P.c, rc);
            sum += m;
            if (!(m > 0.0)) continue;
            last = v0 + e;
            if (first == 0x7fffffff && sum > t) first = v0 + e;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            first = min(first, __shfl_xor_sync(0xffffffffu, first, off));
            last = max(last, __shfl_xor_sync(0xffffffffu, last, off));
        }
        if (lane == 0) drawn = first != 0x7fffffff ? first : max(last, 0);
    }
    team_sync<T>();
    return drawn;
}

// The extra token of a sequence, and what the sequence puts out, by the first T threads of the block that brought the last item of
// the row that it is drawn from, `unit`, once that row's region masses are all there.  `lead`: entries of region 0 before the row.
// Its end is the call's where the sweep is short, and what it consists of is round trips and sums that wait for one another; so many
// threads do it, a region or two to a thread and then a few entries of one (how many: rule and figures at launch_sweeps, host).
// From the last item to the end of the call 4 us; by one warp with sixteen regions and entries to a lane, one after the other,
// 7.5.  Calls, one warp / 256 threads, normal logits, back to back in one run: 16 sequences, 5 tokens, 50 257 bf16 entries 25.1 / 19.3 us,
// 16, 5, 65 536 20.8 / 18.4, 12, 4, 128 256 fp32 23.5 / 21.5, error feedback 64, 4, 151 936 bf16 51.2 / 49.2.  (Run once beforehand
// by blocks that wait anyway, so that its instructions are there: slower, 52.6 for 51.2 as it was then.)
template <int DT, int T>
__device__ __noinline__ void sweep_draw(const Params& P, int unit, int lead) {
    using E = Elem<DT>;
    constexpr int kEntries = kRegionVecs * E::VEC, PER = kEntries / T;
    static_assert(SD_MAX_K < T, "a thread for every token");
    __shared__ double sums[2][T / 32];
    __shared__ double prefix_sh;
    __shared__ int owner[2], found, last_mass;
    const int tid = threadIdx.x, k = P.k, NR = P.NR;
    const int b = unit / (k + 1), n = unit - b * (k + 1);
    const bool bonus = n == k;
    if (!SD_IN(unit, P.B * (k + 1), 23)) return;
    const float* const rs = P.region_sums + (size_t)unit * NR;
    const size_t offT = (size_t)unit * P.V, offD = (size_t)(b * k + (bonus ? 0 : n)) * P.V;
    // (everything that depends on nothing, at once)
    const float4 rcv = __ldcg(reinterpret_cast<const float4*>(P.rowc + unit));
    const RowConst rc{rcv.x, rcv.y, rcv.z, rcv.w};
    const double uk = (double)P.u[b * (k + 1) + k];
    const int32_t x = tid < n ? P.x[b * k + tid] : -1;
    uint32_t word = 0, flags = 0;
    if (tid == 0) {
        word = __ldcg(P.wstatus + b) | (__ldcg(P.sticky) != 0 ? kStatusTimeout : 0u);
        owner[0] = owner[1] = found = 0x7fffffff;
        last_mass = -1;
    }
    const int per = (NR + T - 1) / T, j0 = tid * per, j1 = min(NR, j0 + per);
    const int mode = bonus ? 1 : 0;
    int y = 0;
    // (the first two regions of a thread stay in registers: rows of up to 512 regions)
    float held[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) held[q] = j0 + q < j1 ? __ldcg(rs + j0 + q) : 0.f;
    double all, mine = (double)held[0] + (double)held[1];
    for (int j = j0 + 2; j < j1; ++j) mine += (double)__ldcg(rs + j);
    const double before = team_sums_before<T>(mine, sums[0], &all);
    const double t = uk * all;
    if (!(all > 0.0) || !isfinite(all)) {                          // (the same for every thread)
        flags |= bonus ? SD_STATUS_BAD_ROW : SD_STATUS_ZERO_RESIDUAL;
        if (!bonus) y = sweep_draw_from_p<DT, T>(P, rc, offT, uk, lead);
    } else {
        // the first region whose running sum exceeds t, or (rounding pushed u * R to the total) the last with mass
        if (mine > 0.0 && before + mine > t) atomicMin(&owner[0], tid);
        if (mine > 0.0) atomicMax(&last_mass, tid);
        team_sync<T>();
        const bool past_end = owner[0] == 0x7fffffff;
        if (tid == (past_end ? last_mass : owner[0])) {
            int at = -1;
            double run = before;
            for (int j = j0; j < j1; ++j) {
                const double m = j == j0 ? (double)held[0] : j == j0 + 1 ? (double)held[1] : (double)__ldcg(rs + j);
                if (!(m > 0.0)) continue;
                at = j;
                if (!past_end && run + m > t) break;
                run += m;
            }
            found = max(at, 0);
            prefix_sh = run;
        }
        team_sync<T>();
        const int region = found;
        const double prefix = past_end ? 0.0 : prefix_sh;
        if (tid == 0) last_mass = -1;
        // the same among the region's entries, recomputed as they were
        float m[PER];
        const int v0 = region * kEntries + tid * PER - lead;
        mine = 0.0;
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const bool in = v0 + e >= 0 && v0 + e < P.V && SD_IN(region, NR, 24);
            const float tl = in ? E::load(P.T, offT + v0 + e) : -INFINITY, dl = in && mode == 0 ? E::load(P.D, offD + v0 + e) : -INFINITY;
            m[e] = in ? mass_of(tl, dl, P.c, rc, mode) : 0.f;
            mine += (double)m[e];
        }
        double region_all;
        const double inside = prefix + team_sums_before<T>(mine, sums[1], &region_all);
        if (!past_end && mine > 0.0 && inside + mine > t) atomicMin(&owner[1], tid);
        if (mine > 0.0) atomicMax(&last_mass, tid);
        team_sync<T>();
        // (region sum and re-summed entries may disagree in the last bits: the last entry with mass then, too)
        const bool to_last = owner[1] == 0x7fffffff;
        if (tid == (to_last ? last_mass : owner[1])) {
            int at = -1;
            double run = inside;
#pragma unroll
            for (int e = 0; e < PER; ++e) {
                if (m[e] > 0.f && (to_last || at < 0 || !(run > t))) at = v0 + e;     // (the first behind which the sum exceeds t)
                run += (double)m[e];
            }
            found = max(at, 0);
        }
        if (tid == 0 && last_mass < 0) found = 0;
        team_sync<T>();
        y = found;
    }
    if (tid == 0) {
        P.accept_len[b] = n;
        const uint32_t st = word | flags;
        if (P.status && st) atomicOr(P.status + b, st);
        P.wstatus[b] = 0;               // ready for the next call
    }
    if (tid <= k && SD_IN(b * (k + 1) + tid, P.B * (k + 1), 25)) P.tokens[b * (k + 1) + tid] = tid == n ? y : x;
}

// Sums over a whole row of the second sweep, by one warp of the block that brought the row's last item: hint error,
// acceptance probability.
template <bool HINT>
__device__ __noinline__ void sweep_row_sums(const Params& P, const Sweep& S, int unit, size_t d_row) {
    const int lane = threadIdx.x & 31;
    if (!SD_IN(unit, total_units<false>(P), 23) || !SD_IN(d_row, (long long)P.B * P.k, 21)) return;
    if (HINT) {
        // the items' shares in their order
        double e = 0.0;
        const double* hp = P.hint_part + (size_t)unit * P.hint_stride;
        for (int i = 0; i < S.slices; ++i) e += __ldcg(hp + i);
        if (lane == 0) P.hint_err[d_row] = (float)e;
    }
    if (S.all_rows) {
        // diagnostic: acceptance probability 1 - sum max(0,p-q) of the position
        const float* rs = P.region_sums + (size_t)unit * P.NR;
        double part = 0.0;
        for (int j = lane; j < P.NR; j += 32) part += (double)__ldcg(rs + j);
        const double R = warp_sum(part) * (double)P.tau;
        if (lane == 0) P.acc_prob[d_row] = (float)(1.0 - R);
    }
}

// One block per item.  The first S.draw_blocks blocks take the rows that are drawn from (so that the draws,
// chains of dependent reads, are over long before the sweep is); the rest all other pair rows, from the
// last item of the first sweep backwards.  (Blocks for bonus rows, which would only find nothing to do: 32 sequences, 8
// tokens, 128 256 bf16 entries 57.7 us, without 57.4.)
template <int DT, int MODE, bool RAGGED, bool FINE>
__global__ void __launch_bounds__(kSweepThreads, MODE == kSweepHint || RAGGED ? 4 : 6)
sd_sweep_grad_kernel(const __grid_constant__ Params P, const __grid_constant__ Sweep S) {
    using E = Elem<DT>;
    using ET = typename E::type;
    constexpr bool ERR = MODE == kSweepErrors, HINT = MODE == kSweepHint;
    __shared__ float hpart[kSweepWarps];
    __shared__ int is_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool draws = (int)blockIdx.x < S.draw_blocks;
    int unit, slice, b, regions = S.draw_regions, slices = S.draw_slices;
    if (draws) {
        b = (int)blockIdx.x / S.draw_slices;
        slice = (int)blockIdx.x - b * S.draw_slices;
        unit = 0;
    } else {
        // FINE: of the last rows the large items, then of the first ones the small
        int id = (int)(gridDim.x - 1u - blockIdx.x), from = 0, rows = P.B * P.k;
        regions = S.regions;
        slices = S.slices;
        if constexpr (FINE) {
            if (id < S.fine_rows * S.fine_slices) {
                rows = S.fine_rows;
                regions = S.fine_regions;
                slices = S.fine_slices;
            } else {
                from = S.fine_rows;
                id -= from * S.fine_slices;
                rows -= from;
            }
        }
        slice = id / rows;
        const int row = from + id - slice * rows;
        b = row / P.k;
        unit = row + b;
    }
    await_previous_kernel();
    launch_dependents();

    if (!SD_IN(b, P.B, 22) || !SD_IN(unit, total_units<false>(P), 20)) return;
    if (!SD_IN(slice, slices, 20)) return;
    // (both loads under way together: of a block's chain of round trips this is one less)
    RowConst rc = P.rowc[unit];
    const int n = P.accept[b * P.k];
    if (draws) {
        unit = b * (P.k + 1) + n;
        if (!SD_IN(unit, total_units<false>(P), 20)) return;
        rc = P.rowc[unit];
    }
    const int i = unit - b * (P.k + 1);
    if (!draws && i == n) return;                     // the first blocks have it
    // (not from the unit: another division, on the way of every block; 450 sequences, 16 tokens, 1 000 bf16 entries 48.0 -> 45.2 us)
    const bool bonus = draws && n == P.k;
    const UnitRef ur{b, i, 0, bonus, (size_t)unit, (size_t)b * P.k + (bonus ? 0 : i)};
    const int v0 = (slice * regions + warp) * kRegionVecs;
    float herr = 0.f;
    float* const rsum = P.region_sums + (size_t)unit * P.NR + slice * regions + warp;
    const bool masses = draws || HINT || S.all_rows;
    if constexpr (RAGGED) {
        const RowFrame<DT> f = row_frame<DT>(P, ur);
        int v1 = min((slice + 1) * regions, P.NR) * kRegionVecs;
        if (!SD_IN(ur.t_row, (long long)P.B * (P.k + 1), 12) || !SD_IN(ur.d_row, (long long)P.B * P.k, 12)) v1 = 0;
        if (v0 < v1 && !SD_IN(v0 / kRegionVecs + (v1 - 1 - v0) / kSweepStep * kSweepWarps, P.NR, 13)) v1 = 0;
        ET* const grow = (P.grad && !ur.bonus) ? reinterpret_cast<ET*>(P.grad) + ur.d_row * P.V : nullptr;
        if (ur.bonus)    ragged_pass2<DT, true, true>(f, P.V, v0, v1, nullptr, rsum, lane, P.c, rc);
        else if (masses) ragged_pass2<DT, false, true>(f, P.V, v0, v1, grow, rsum, lane, P.c, rc);
        else             ragged_pass2<DT, false, false>(f, P.V, v0, v1, grow, nullptr, lane, P.c, rc);
    } else {
        int nvec = min((slice + 1) * regions * kRegionVecs, P.V / E::VEC) - v0;
        if (nvec > 0 && !SD_IN((long long)(v0 + nvec) * E::VEC - 1, P.V, 12)) nvec = 0;
        if (!SD_IN(ur.t_row, (long long)P.B * (P.k + 1), 12) || !SD_IN(ur.d_row, (long long)P.B * P.k, 12)) nvec = 0;
        if (nvec > 0 && !SD_IN(v0 / kRegionVecs + (nvec - 1) / kSweepStep * kSweepWarps, P.NR, 13)) nvec = 0;
        const size_t offD = ur.d_row * P.V + (size_t)v0 * E::VEC;
        const size_t offG = ERR ? (size_t)b * P.V + (size_t)v0 * E::VEC : offD;
        const uint4* const gT = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + ur.t_row * P.V) + v0;
        const uint4* const gD = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.D) + offD);
        ET* const gdst = (P.grad && !ur.bonus) ? reinterpret_cast<ET*>(P.grad) + offG : nullptr;
        const uint64_t policy = policy_discard();
        if (ur.bonus) {
            sweep_pass2<DT, true, false, true>(gT, gD, nullptr, nullptr, rsum, nvec, lane, P.c, policy, rc, herr);
            if (ERR && P.grad) {
                // no error position: a zero row
                uint4* z = reinterpret_cast<uint4*>(reinterpret_cast<ET*>(P.grad) + offG);
                for (; nvec > 0; nvec -= kSweepStep, z += kSweepStep) {
#pragma unroll
                    for (int g = 0; g < kRegionRows; ++g)
                        if (g * 32 + lane < nvec) __stcs(z + g * 32 + lane, make_uint4(0u, 0u, 0u, 0u));
                }
            }
        } else if (masses) {
            const uint4* const gH = HINT ? reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.hint) + offD) : nullptr;
            sweep_pass2<DT, false, HINT, true>(gT, gD, gH, gdst, rsum, nvec, lane, P.c, policy, rc, herr);
        } else {
            sweep_pass2<DT, false, false, false>(gT, gD, nullptr, gdst, nullptr, nvec, lane, P.c, policy, rc, herr);
        }
    }
    if (!masses) return;
    if constexpr (HINT) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) herr += __shfl_xor_sync(0xffffffffu, herr, off);
        if (lane == 0) hpart[warp] = herr;
    }
    __syncthreads();
    if (!draws && warp != 0) return;                  // (of the drawn rows, the block that brings the last item draws)
    if (tid == 0) {
        if (HINT && !ur.bonus) {
            // this item's share of the row's hint error: the warps' shares in their order, in fp64
            double e = 0.0;
            for (int w = 0; w < kSweepWarps; ++w) e += (double)hpart[w];
            if (SD_IN(slice, P.hint_stride, 27)) P.hint_part[(size_t)unit * P.hint_stride + slice] = e;
        }
        is_last = SD_IN(unit, total_units<false>(P), 28) && count_up(S.arrived + unit, 1u, (uint32_t)slices);
        if (is_last) S.arrived[unit] = 0;
    }
    if (draws) __syncthreads();
    else __syncwarp();
    if (!is_last) return;
    if ((HINT || S.all_rows) && !ur.bonus && warp == 0) sweep_row_sums<HINT>(P, S, unit, ur.d_row);
    if (!draws || tid >= S.draw_threads) return;
    const int lead = RAGGED ? row_frame<DT>(P, ur).lead : 0;
    if (S.draw_threads == kSweepThreads) sweep_draw<DT, kSweepThreads>(P, unit, lead);
    else                                 sweep_draw<DT, kSweepThreads / 2>(P, unit, lead);
}

}  // namespace sdv
