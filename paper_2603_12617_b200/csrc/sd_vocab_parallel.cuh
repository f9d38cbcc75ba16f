// The step for logits that are sharded along the vocabulary, as a tensor-parallel output layer
// leaves them (the paper's deployment spreads a model over four GPUs): rank g of G holds the
// columns [v_offset, v_offset + Vs) of every logit row.  A softmax needs every column, so the
// step falls into three local phases with two small exchanges between them:
//
//   phase 1  sd_vp_stats_kernel   per row: softmax sums of the shard relative to integer
//                                 references (a PartialStats), and the logits of the drafted
//                                 token if this shard holds it              -> 48 bytes per row
//   exchange all-gather of the records of all ranks
//   phase 2  sd_vp_rows_kernel    per sequence: the G records of every row merged in rank order
//                                 (exact powers of two, fp64 sums: every rank gets the same bits),
//                                 row constants, KL loss, rejection tests, accept length
//            sd_vp_grad_kernel    second sweep over the shard: the gradient's columns of every
//                                 row, and the masses of the sampling regions of the one row per
//                                 sequence that the extra token is drawn from; the last block of
//                                 that row: this shard's share of its mass, and of the mass
//                                 of p_n (the fallback of a residual without mass)        -> 16 bytes
//   exchange all-gather of the shares
//   phase 3  sd_vp_draw_kernel    per sequence: exclusive scan of the shares in rank order; the rank
//                                 whose interval holds u_k * total searches its own regions and
//                                 writes the token (global index), the others write -1
//   exchange element-wise maximum of the token arrays (the caller's all-reduce)
//
// The arithmetic is that of the single-GPU kernels (same element functions, same merging), so the
// results meet the same bars against the oracle.  Each logit is read from HBM twice here: the
// exchange between the passes is a round trip through the host's collective, and a shard's batch
// does not stay in L2 meanwhile.
#pragma once

#include "sd_kernels.cuh"
#include "sd_sweep.cuh"

namespace sdv {

constexpr int kVpThreads = kSweepThreads;
constexpr int kVpWarps = kVpThreads / 32;

// What a rank tells the others about its shard of one row.
struct __align__(16) VpRecord {
    PartialStats st;         // 32 bytes
    float tx, dx;            // logits of the drafted token (target, draft) if this shard holds it
    uint32_t has_token;      // 1 if it does
    uint32_t pad;
};
static_assert(sizeof(VpRecord) == 48, "record layout is part of the ABI");

struct VpParams {
    const void* T;           // [B,k+1,Vs]
    const void* D;           // [B,k,Vs]
    const int32_t* x;        // [B,k] global token ids
    const float* u;          // [B,k+1]
    int B, k, Vs, v_offset, V_total;
    int G, rank;
    float c, tau;
    double inv_tau;
    int NR;                  // sampling regions per shard row (kRegionVecs vectors each)
    VpRecord* records;       // phase 1 out: [B*(k+1)]
    const VpRecord* all;     // phase 2 in: [G][B*(k+1)]
    int32_t* accept_len;     // [B]
    float* loss;             // [B,k] or null
    void* grad;              // [B,k,Vs] or null
    uint32_t* status;        // [B] or null
    double* local_mass;      // [B][2]: share of the residual (or bonus) mass, share of the mass of p_n
    const double* all_mass;  // phase 3 in: [G][B][2]
    int32_t* tokens;         // [B,k+1]
    // workspace
    RowConst* rowc;          // [B*(k+1)]
    float* region_sums;      // [B][2][NR]: regions of the row the extra token is drawn from: masses of the
                             // residual (or bonus row), and of p_n (what a residual without mass falls back to)
};

// ---- phase 1 -------------------------------------------------------------------------------
// A cluster of C blocks per row (as many as leave all of them resident: a warp's time is a chain of round trips, one
// per region), its warps take the row's regions in turn, with the loop of the single-GPU first sweep (a
// maximum for every two vectors and a test for masked entries took 18.0 us on 320 rows of 37 984 bf16 entries,
// one block of eight warps per row 15.7; ten or twelve blocks an SM, with fewer registers, no less, and fp32 rows a tenth more).
// PAIRS: a warp's regions two at a time (fp32 rows; rule and figures: sd_vp_partial, host).
// Every region raises the references: with those of a warp's first region alone the error of fp32
// gradients against 64 bits doubled.  With a vote whether any entry is above them that costs nothing there
// (1792 rows of 32 064 entries 42.0 -> 44.0; raised without looking 45.0).
constexpr int kVpStatsWarps = 4;
constexpr int kVpStatsThreads = kVpStatsWarps * 32;
constexpr int kVpMaxCluster = 8;
template <int DT, bool PAIRS>
__global__ void __launch_bounds__(kVpStatsThreads, 8) sd_vp_stats_kernel(const VpParams P) {
    using E = Elem<DT>;
    using ET = typename E::type;
    constexpr int VEC = E::VEC;
    __shared__ PartialStats part[kVpMaxCluster * kVpStatsWarps];     // of the cluster's first block: every warp's
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    if (C > 1) cluster_arrive();                                     // (waited for before the first remote store)
    await_previous_kernel();
    launch_dependents();
    const int unit = (int)blockIdx.x / C;
    const int K1 = P.k + 1;
    const int b = unit / K1, i = unit - b * K1;
    const bool bonus = (i == P.k);
    const int tid = threadIdx.x, lane = tid & 31, slot = rank * kVpStatsWarps + (tid >> 5), slots = C * kVpStatsWarps;
    const bool reports = rank == 0 && tid == 0;
    const uint4* Trow = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + (size_t)unit * P.Vs);
    const uint4* Drow = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.D) + (size_t)(b * P.k + (bonus ? 0 : i)) * P.Vs);
    const int NV = P.Vs / VEC;

    // (the drafted token's logits are asked for first: two dependent reads that the sweep hides)
    float tx = 0.f, dx = 0.f;
    uint32_t has_token = 0;
    if (reports && !bonus) {
        const int xg = P.x[b * P.k + i] - P.v_offset;
        if (xg >= 0 && xg < P.Vs) {
            has_token = 1;
            tx = E::load(P.T, (size_t)unit * P.Vs + xg);
            dx = E::load(P.D, (size_t)(b * P.k + i) * P.Vs + xg);
        }
    }
    Pass1State ps;
    ps.RT = ps.RD = kEmptyRef;
    ps.ls.init();
    const int w0 = slot * kRegionVecs;
    const uint64_t policy = policy_normal();     // what fits stays in L2 for the second sweep
    const int nvec = SD_IN(unit, P.B * K1, 60) ? NV - w0 : 0;
    const int step = slots * kRegionVecs;
    if constexpr (PAIRS) {
        if (bonus) sweep_pass1_pairs<DT, true>(Trow + w0, Drow + w0, nvec, step, lane, P.c, policy, ps);
        else       sweep_pass1_pairs<DT, false>(Trow + w0, Drow + w0, nvec, step, lane, P.c, policy, ps);
    } else {
        if (bonus) sweep_pass1<DT, true, true>(Trow + w0, Drow + w0, nvec, step, lane, P.c, policy, ps);
        else       sweep_pass1<DT, false, true>(Trow + w0, Drow + w0, nvec, step, lane, P.c, policy, ps);
    }
    __syncwarp();
    if (C > 1) {
        cluster_wait();
        warp_post_lanes(ps.ls, ps.RT, ps.RD, lane, cluster.map_shared_rank(&part[slot], 0));
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    } else {
        warp_post_lanes(ps.ls, ps.RT, ps.RD, lane, &part[slot]);
        __syncthreads();
    }
    if (rank == 0 && tid < 32) {
        VpRecord r;
        r.st = warp_merge_lanes(lane < slots ? part[lane] : empty_partial());
        r.tx = tx;
        r.dx = dx;
        r.has_token = has_token;
        r.pad = 0;
        if (lane == 0 && SD_IN(unit, P.B * K1, 60)) P.records[unit] = r;
    }
}

// ---- phase 2 -------------------------------------------------------------------------------
// One block per sequence, one warp per row (up to kRowsMaxWarps of them at a time), one lane per rank: merge of the G
// records of the row in a fixed order, row constants, loss, rejection test; then the accept length.  Every rank
// computes the same bits.
__global__ void __launch_bounds__(kRowsMaxWarps * 32) sd_vp_rows_kernel(const VpParams P) {
    __shared__ uint8_t accepted[SD_MAX_K + 1];
    __shared__ uint32_t flags_sh;
    await_previous_kernel();
    launch_dependents();
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = (int)blockDim.x >> 5;
    const int K1 = P.k + 1;
    if (threadIdx.x == 0) flags_sh = 0;
    __syncthreads();
    for (int i = warp; i < K1; i += warps) {
        const int unit = b * K1 + i;
        const bool bonus = (i == P.k);
        const size_t rows = (size_t)P.B * K1;
        const int xg = bonus ? 0 : P.x[b * P.k + i];
        const float u = P.u[b * K1 + i];
        PartialStats st = empty_partial();
        float tx = 0.f, dx = 0.f;
        bool have = false;
        for (int g0 = 0; g0 < P.G; g0 += 32) {
            PartialStats part = empty_partial();
            bool has = false;
            float t = 0.f, d = 0.f;
            if (g0 + lane < P.G) {
                const VpRecord r = P.all[(size_t)(g0 + lane) * rows + unit];
                part = r.st;
                has = r.has_token != 0;
                t = r.tx;
                d = r.dx;
            }
            part = warp_merge_lanes(part);
            if (g0 == 0) {
                st = part;
            } else {
                const float RT = fmaxf(st.RT, part.RT), RD = fmaxf(st.RD, part.RD);
                const PartialStats a = rescaled(st, RT, RD), c = rescaled(part, RT, RD);
                st.RT = RT; st.RD = RD;
                st.sT = a.sT + c.sT; st.sD = a.sD + c.sD; st.w = a.w + c.w;
            }
            const unsigned m = __ballot_sync(0xffffffffu, has);
            if (m && !have) {
                have = true;
                tx = __shfl_sync(0xffffffffu, t, __ffs(m) - 1);
                dx = __shfl_sync(0xffffffffu, d, __ffs(m) - 1);
            }
        }
        const RowLogs logs = warp_row_logs(st);
        if (lane != 0) continue;
        const RowConst rc = row_constants_of(P.inv_tau, bonus, st);
        P.rowc[unit] = rc;
        uint32_t flags = 0;
        const bool okT = (st.sT > 0.0) && isfinite(st.sT);
        const bool okD = bonus || ((st.sD > 0.0) && isfinite(st.sD));
        if (!okT || !okD) flags |= SD_STATUS_BAD_ROW;
        bool acc = true;
        if (!bonus) {
            const double l2ST = logs.T, l2SD = logs.D;
            if (P.loss) P.loss[b * P.k + i] = (float)(0.6931471805599453 * (st.w / st.sT - l2ST + l2SD));
            acc = false;
            if (xg < 0 || xg >= P.V_total || !have) {
                flags |= SD_STATUS_BAD_TOKEN;
            } else if (okT && okD) {
                const double dtx = (double)tx, ddx = (double)dx;
                double rho;
                if (ddx == -INFINITY) {
                    rho = (dtx == -INFINITY) ? 0.0 : INFINITY;
                } else {
                    const double l2p = (dtx * (double)P.c - (double)st.RT) - l2ST;
                    const double l2q = (ddx * (double)P.c - (double)st.RD) - l2SD;
                    rho = exp2(l2p - l2q);
                }
                acc = (double)u < (rho < 1.0 ? rho : 1.0);
            }
        }
        accepted[i] = acc ? 1 : 0;
        if (flags) atomicOr(&flags_sh, flags);
    }
    __syncthreads();
    if (warp != 0) return;
    int n = P.k;
    for (int i0 = 0; i0 < P.k; i0 += 32) {
        const unsigned m = __ballot_sync(0xffffffffu, i0 + lane < P.k && !accepted[i0 + lane]);
        if (m) { n = i0 + __ffs(m) - 1; break; }
    }
    if (lane == 0) {
        P.accept_len[b] = n;
        if (P.status) P.status[b] = flags_sh;
        // until the gradient kernel has the masses, their place counts the blocks that have written theirs
        *reinterpret_cast<uint32_t*>(P.local_mass + (size_t)b * 2) = 0;
    }
}

// Second sweep over the shard: one block per (row, slice of sampling regions).  Gradient of every
// pair row; masses of the regions of row n_b of every sequence (the bonus row when n_b = k); and, by the block that
// brings that row's last slice, this shard's share of the row's mass (fixed order, fp64).  Rows that are not drawn
// from skip their masses.
template <int DT>
__global__ void __launch_bounds__(kVpThreads, 6) sd_vp_grad_kernel(const VpParams P, const int slices, const int regions) {
    using E = Elem<DT>;
    using ET = typename E::type;
    constexpr int VEC = E::VEC;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int unit = (int)blockIdx.x / slices, sl = (int)blockIdx.x - unit * slices;
    const int K1 = P.k + 1;
    const int b = unit / K1, i = unit - b * K1;
    const bool bonus = (i == P.k);
    launch_dependents();
    await_previous_kernel();
    const int n = P.accept_len[b];
    const bool draws = (i == n);                     // the extra token comes from this row
    if (bonus && !draws) return;                     // a bonus row that is not drawn from has nothing to do
    if (!draws && !P.grad) return;
    const RowConst rc = P.rowc[unit];
    const uint4* Trow = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.T) + (size_t)unit * P.Vs);
    const uint4* Drow = reinterpret_cast<const uint4*>(reinterpret_cast<const ET*>(P.D) + (size_t)(b * P.k + (bonus ? 0 : i)) * P.Vs);
    ET* Grow = (P.grad && !bonus) ? reinterpret_cast<ET*>(P.grad) + (size_t)(b * P.k + i) * P.Vs : nullptr;
    const int NV = P.Vs / VEC;
    float* rsum = P.region_sums + (size_t)b * 2 * P.NR;
    const int r0 = sl * regions, r1 = min(P.NR, r0 + regions);
    if (!draws) {
        const int v0 = (r0 + warp) * kRegionVecs;
        int nvec = min(r1 * kRegionVecs, NV) - v0;
        if (nvec > 0 && (!SD_IN((long long)(v0 + nvec) * VEC - 1, P.Vs, 61) || !SD_IN(unit, P.B * K1, 62))) nvec = 0;
        float unused = 0.f;
        sweep_pass2<DT, false, false, false>(Trow + v0, Drow + v0, nullptr, Grow + (size_t)v0 * VEC, nullptr, nvec, lane, P.c,
                                             policy_discard(), rc, unused);
        return;
    }
    for (int r = r0 + warp; r < r1; r += kVpWarps) {
        const int v0 = r * kRegionVecs;
        const int nv = min(kRegionVecs, NV - v0);
        if (!SD_IN((long long)(v0 + nv) * VEC - 1, P.Vs, 61) || !SD_IN(unit, P.B * K1, 62)) continue;
        uint4 rt[kRegionRows], rd[kRegionRows];
#pragma unroll
        for (int g = 0; g < kRegionRows; ++g) {
            const int vi = g * 32 + lane;
            rt[g] = vi < nv ? __ldcs(Trow + v0 + vi) : E::masked();
            rd[g] = (!bonus && vi < nv) ? __ldcs(Drow + v0 + vi) : E::masked();
        }
        const float mass = bonus ? pass2_region<DT, true>(rt, rd, nv, lane, P.c, rc, nullptr)
                                 : pass2_region<DT, false>(rt, rd, nv, lane, P.c, rc, Grow ? Grow + (size_t)v0 * VEC : nullptr);
        {
            // mass of p_n in the region as well: a rejection whose residual has no mass draws from p_n
            float pm = 0.f;
            if (!bonus) {
#pragma unroll
                for (int g = 0; g < kRegionRows; ++g) {
                    float tv[VEC];
                    E::unpack(rt[g], tv);
                    if (g * 32 + lane < nv) {
#pragma unroll
                        for (int e = 0; e < VEC; ++e) pm += prob_elem(tv[e], P.c, rc);
                    }
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) pm += __shfl_xor_sync(0xffffffffu, pm, off);
            }
            if (lane == 0) { rsum[r] = mass; rsum[P.NR + r] = pm; }
        }
    }
    __shared__ int is_last;
    __syncthreads();
    if (tid == 0) is_last = count_up(reinterpret_cast<uint32_t*>(P.local_mass + (size_t)b * 2), 1u, (uint32_t)slices);
    __syncthreads();
    if (!is_last || warp > 1) return;
    // (one warp to each of the two masses)
    const int per = (P.NR + 31) / 32;
    const int j0 = min(P.NR, lane * per), j1 = min(P.NR, j0 + per);
    const float* const rs = rsum + (size_t)warp * P.NR;
    double mine = 0.0;
    for (int j = j0; j < j1; ++j) mine += (double)__ldcg(rs + j);
    const double incl = warp_inclusive_scan(mine);
    if (lane == 31) P.local_mass[(size_t)b * 2 + warp] = incl;
}

// ---- phase 3 -------------------------------------------------------------------------------
// One block of T threads per sequence.  Shares in rank order: the first rank whose running sum exceeds
// u_k * total owns the draw (the last rank with mass, if rounding leaves none); its block searches as the single-GPU
// draw does (sweep_draw), with the mass of the ranks before it in front.  128 threads, 64 where there are more than four blocks to
// an SM.  This kernel alone, the warp that drew once / 64 / 128 / 256 threads, us: 64 sequences, 37 984 bf16 entries 4.6 / 4.3 / 3.8 /
// 3.8, 512 of 8 000 5.1 / 4.4 / 4.2 / 5.9, 1000 of 16 000 4.8 / 4.4 / 5.1 / 6.5; fp32 256 of 19 000 3.8 / 4.1 / 3.7 / 3.9, 512 of 8 000 4.2 / 4.2 / 4.2 /
// 5.8, 1000 of 512 3.8 / 4.0 / 5.5 / 6.4, 2000 of 256 4.8 / 5.5 / 6.5 / 9.8.
template <int DT, int T>
__global__ void __launch_bounds__(T) sd_vp_draw_kernel(const VpParams P) {
    using E = Elem<DT>;
    constexpr int kEntries = kRegionVecs * E::VEC, PER = kEntries / T;
    __shared__ double sums[2][T / 32];
    __shared__ double prefix_sh;
    __shared__ int owner_sh[2], found, last_mass;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int k = P.k, K1 = k + 1;
    await_previous_kernel();
    launch_dependents();
    // everything that does not depend on where the draw falls is asked for at once: the block's time is round trips
    // (the caller's memory: a length that phase 2 cannot have written leads to no row but the sequence's own)
    const int n = min(max(P.accept_len[b], 0), k);
    const double uk = (double)P.u[b * K1 + k];
    const int32_t x = tid < k ? P.x[b * k + tid] : -1;
    double2 mass = make_double2(0.0, 0.0);
    if (lane < P.G) {
        const double* const m = P.all_mass + ((size_t)lane * P.B + b) * 2;
        mass = make_double2(m[0], m[1]);
    }
    const int per = (P.NR + T - 1) / T, j0 = min(P.NR, tid * per), j1 = min(P.NR, j0 + per);
    const float* rs = P.region_sums + (size_t)b * 2 * P.NR;
    float held = j0 < j1 ? rs[j0] : 0.f;
    if (tid == 0) {
        owner_sh[0] = owner_sh[1] = 0x7fffffff;
        found = 0;
        last_mass = -1;
    }
    const bool bonus = (n == k);
    const int unit = b * K1 + n;
    const RowConst rc = P.rowc[unit];
    // rank g's shares (every warp finds the same)
    const auto share = [&](int g, int which) {
        if (P.G > 32) return P.all_mass[((size_t)g * P.B + b) * 2 + which];
        return __shfl_sync(0xffffffffu, which ? mass.y : mass.x, g);
    };
    uint32_t flags = 0;
    int which = 0;
    double total = 0.0;
    for (int g = 0; g < P.G; ++g) total += share(g, 0);
    if (!bonus && !(total > 0.0)) {
        // a rejection whose residual has no mass on any rank (q = p and a forced rejection): the extra
        // token comes from p_n, and the status says so
        flags |= SD_STATUS_ZERO_RESIDUAL;
        which = 1;
        total = 0.0;
        for (int g = 0; g < P.G; ++g) total += share(g, 1);
        rs += P.NR;
        held = j0 < j1 ? rs[j0] : 0.f;
    }
    const int mode = bonus ? 1 : (which ? 2 : 0);
    const double t = uk * total;
    int owner = -1, last_with_mass = -1;
    double ahead = 0.0, run = 0.0;
    for (int g = 0; g < P.G; ++g) {
        const double m = share(g, which);
        if (m > 0.0) last_with_mass = g;
        if (owner < 0 && run + m > t) { owner = g; ahead = run; }
        run += m;
    }
    bool past_end = false;
    if (owner < 0) { owner = last_with_mass; past_end = true; }
    int y = -1;
    if (!(total > 0.0) || !isfinite(total)) {
        // no mass anywhere (a row without a usable denominator): the first entry of the vocabulary
        // stands in, and the status says so
        flags |= SD_STATUS_BAD_ROW;
        if (P.rank == 0) y = 0;
    } else if (owner == P.rank) {                     // (the same for every thread)
        const size_t offT = (size_t)unit * P.Vs, offD = (size_t)(b * k + (bonus ? 0 : n)) * P.Vs;
        double mine = (double)held, all;
        for (int j = j0 + 1; j < j1; ++j) mine += (double)rs[j];
        const double before = ahead + team_sums_before<T>(mine, sums[0], &all);
        if (!past_end && mine > 0.0 && before + mine > t) atomicMin(&owner_sh[0], tid);
        if (mine > 0.0) atomicMax(&last_mass, tid);
        team_sync<T>();
        const bool to_last = owner_sh[0] == 0x7fffffff;      // (rounding: the last region of this shard that holds mass)
        if (tid == (to_last ? last_mass : owner_sh[0])) {
            int at = j0;
            double r2 = before;
            for (int j = j0; j < j1; ++j) {
                const double m = j == j0 ? (double)held : (double)rs[j];
                if (!(m > 0.0)) continue;
                at = j;
                if (!to_last && r2 + m > t) break;
                r2 += m;
            }
            found = at;
            prefix_sh = r2;
        }
        team_sync<T>();
        const int region = found;
        const double prefix = to_last ? 0.0 : prefix_sh;
        if (tid == 0) last_mass = -1;
        float m[PER];
        const int v0 = region * kEntries + tid * PER;
        mine = 0.0;
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const bool in = v0 + e < P.Vs && SD_IN(region, P.NR, 63);
            const float tl = in ? E::load(P.T, offT + v0 + e) : -INFINITY, dl = in && mode == 0 ? E::load(P.D, offD + v0 + e) : -INFINITY;
            m[e] = in ? mass_of(tl, dl, P.c, rc, mode) : 0.f;
            mine += (double)m[e];
        }
        const double inside = prefix + team_sums_before<T>(mine, sums[1], &all);
        if (!to_last && mine > 0.0 && inside + mine > t) atomicMin(&owner_sh[1], tid);
        if (mine > 0.0) atomicMax(&last_mass, tid);
        team_sync<T>();
        const bool last_entry = owner_sh[1] == 0x7fffffff;
        if (tid == (last_entry ? last_mass : owner_sh[1])) {
            int at = -1;
            double r2 = inside;
#pragma unroll
            for (int e = 0; e < PER; ++e) {
                if (m[e] > 0.f && (last_entry || at < 0 || !(r2 > t))) at = v0 + e;     // (the first behind which the sum exceeds t)
                r2 += (double)m[e];
            }
            found = max(at, 0);
        }
        if (tid == 0 && last_mass < 0) found = 0;
        team_sync<T>();
        y = P.v_offset + found;
    }
    if (tid == 0 && flags && P.status) atomicOr(P.status + b, flags);
    for (int i = tid; i <= k; i += T) P.tokens[b * K1 + i] = i < n ? (i == tid ? x : P.x[b * k + i]) : (i == n ? y : -1);
}

}  // namespace sdv
