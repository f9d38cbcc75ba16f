// Greedy verification (Algorithm 1 in the limit tau -> 0; the decoding mode of the paper's
// experiments, Sec. 4.1): a draft token is accepted iff it is the target's argmax of its position,
// and the extra token is the target's argmax at the first mismatch (or at the bonus position).
// Only the target logits are read, once: the kernel is a streaming argmax, bound by HBM.
//
//   sd_greedy_kernel   items are pieces of kGreedyItemVecs 16-byte vectors of a row; every block has a
//                      contiguous run of them, so mostly of one row.  A thread keeps the largest value it has
//                      seen in the row and its first index and asks for the next item's vectors before it
//                      looks at this one's; when the run leaves a row (and at its end) a warp folds its
//                      lanes into one 64-bit key (value in an order-preserving integer form, then the
//                      complement of the index, so that the larger key is the larger value and, among
//                      equals, the smaller index) and applies it to the row's key with one atomicMax whose
//                      result nobody reads.  Warps never wait for one another inside the loop.  A block
//                      that has run out of items takes a ticket; the block with the last ticket reads all
//                      keys, compares them with the draft tokens and writes accept lengths and tokens.
//                      Nobody waits for anybody.  Rows that are not whole vectors are read from the aligned
//                      address before them, their two ends entry by entry.
//
// 288 rows of 128 256 bf16 entries: 22.5 us with one row's item after another and a reduction for each, and a
// last block that read one key after the other; 16.8 us as it is (18.6 before it was launched
// programmatically and took its ticket with one release; 74 MB: 11.3 us at the copy bandwidth, the rest
// is launch, ramp and the last block).
#pragma once

#include "sd_device.cuh"

namespace sdv {

constexpr int kGreedyThreads = 256;
constexpr int kGreedyLoads = 4;                        // vectors of an item per thread: as many again are on their way
constexpr int kGreedyItemVecs = kGreedyLoads * kGreedyThreads;   // 16 KiB of a row
constexpr int kGreedyTailRows = 1024;                  // rows the last block works out at a time (at least SD_MAX_K + 1)

struct GreedyParams {
    const void* T;            // [B,k+1,V]
    const int32_t* x;         // [B,k]
    int B, k, V;
    int items_per_row;
    int32_t* accept_len;      // [B]
    int32_t* tokens;          // [B,k+1]
    int32_t* argmax;          // [B,k+1] or null
    unsigned long long* keys; // [B*(k+1)] zero on entry and zero again on exit
    uint32_t* ticket;         // one word, zero on entry and zero again on exit
};

// Larger value -> larger key; equal values -> smaller index -> larger key.  v is not NaN.
__device__ __forceinline__ unsigned long long greedy_key(float v, int idx) {
    const uint32_t u = __float_as_uint(v + 0.f);                 // -0 becomes +0: equal values, equal keys
    const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)ord << 32) | (uint32_t)(0x7fffffff - idx);
}
__device__ __forceinline__ int greedy_index(unsigned long long key) {
    return key == 0ull ? 0 : 0x7fffffff - (int)(uint32_t)(key & 0xffffffffu);   // untouched key: a row without a finite or +inf entry
}

// Piece `piece` of row `row`: the entry its vector 0 would start at in the row (may be negative), and where the
// row is in memory.
template <int DT> struct GreedyItem {
    int row, piece, e0;
    const typename Elem<DT>::type* rowp;
};
template <int DT>
__device__ __forceinline__ GreedyItem<DT> greedy_item(const GreedyParams& P, int row, int piece) {
    constexpr int VEC = Elem<DT>::VEC;
    GreedyItem<DT> g;
    g.row = row;
    g.piece = piece;
    g.rowp = reinterpret_cast<const typename Elem<DT>::type*>(P.T) + (size_t)row * P.V;
    const int lead = (int)((reinterpret_cast<uintptr_t>(g.rowp) / sizeof(typename Elem<DT>::type)) & (VEC - 1));
    g.e0 = piece * kGreedyItemVecs * VEC - lead;
    return g;
}
// This thread's vectors of an item: whole vectors of the row as they are, the row's ends entry by entry, -inf
// for what is not in the row.
template <int DT>
__device__ __forceinline__ void greedy_fetch(const GreedyItem<DT>& g, int V, int tid, uint4 (&q)[kGreedyLoads]) {
    using E = Elem<DT>;
    constexpr int VEC = E::VEC;
#pragma unroll
    for (int j = 0; j < kGreedyLoads; ++j) {
        const int e = g.e0 + (j * kGreedyThreads + tid) * VEC;
        q[j] = E::masked();
        if (e >= 0 && e + VEC <= V) {
            if (SD_IN(e + VEC - 1, V, 41)) q[j] = __ldcs(reinterpret_cast<const uint4*>(g.rowp + e));
        } else if (e > -VEC && e < V) {
            float v[VEC];
#pragma unroll
            for (int z = 0; z < VEC; ++z) v[z] = (e + z >= 0 && e + z < V) ? E::load(g.rowp, e + z) : -INFINITY;
            q[j] = E::pack(v);               // (bf16 values come back as they were)
        }
    }
}

template <int DT>
__global__ void __launch_bounds__(kGreedyThreads, 4) sd_greedy_kernel(const GreedyParams P) {
    using E = Elem<DT>;
    constexpr int VEC = E::VEC;
    __shared__ int is_last;
    __shared__ int am_sh[kGreedyTailRows], x_sh[kGreedyTailRows];
    await_previous_kernel();
    launch_dependents();
    const int tid = threadIdx.x, lane = tid & 31;
    const int K1 = P.k + 1;
    const long long items = (long long)P.B * K1 * P.items_per_row;
    const long long share = items / gridDim.x, extra = items % gridDim.x;      // the first `extra` blocks have one more
    const long long lo = share * blockIdx.x + min((long long)blockIdx.x, extra);
    const int n_items = (int)(share + (blockIdx.x < extra ? 1 : 0));

    float best = -INFINITY;
    int besti = 0x7fffffff;
    auto flush = [&](int row) {
        unsigned long long key = best > -INFINITY ? greedy_key(best, besti) : 0ull;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, key, off);
            key = o > key ? o : key;
        }
        if (lane == 0 && key != 0ull && SD_IN(row, (long long)P.B * K1, 40)) atomicMax(P.keys + row, key);
        best = -INFINITY;
        besti = 0x7fffffff;
    };
    uint4 q[kGreedyLoads];
    const int row0 = (int)(lo / P.items_per_row);
    GreedyItem<DT> cur = greedy_item<DT>(P, row0, (int)(lo - (long long)row0 * P.items_per_row));
    if (n_items > 0) greedy_fetch<DT>(cur, P.V, tid, q);
    for (int it = 0; it < n_items; ++it) {
        uint4 nq[kGreedyLoads];
        GreedyItem<DT> nx = cur;
        if (it + 1 < n_items) {
            const bool wrap = cur.piece + 1 == P.items_per_row;
            nx = greedy_item<DT>(P, cur.row + (wrap ? 1 : 0), wrap ? 0 : cur.piece + 1);
            greedy_fetch<DT>(nx, P.V, tid, nq);
        }
#pragma unroll
        for (int j = 0; j < kGreedyLoads; ++j) {
            const int e = cur.e0 + (j * kGreedyThreads + tid) * VEC;
            float v[VEC];
            E::unpack(q[j], v);
            // the vector's largest value first: few vectors have one above everything so far
            const float m = tree_max<VEC>(v);
            if (m > best) {
#pragma unroll
                for (int z = 0; z < VEC; ++z)
                    if (v[z] > best) { best = v[z]; besti = e + z; }   // strict: keeps the first index
            }
        }
        if (it + 1 == n_items || nx.row != cur.row) flush(cur.row);
        cur = nx;
#pragma unroll
        for (int j = 0; j < kGreedyLoads; ++j) q[j] = nq[j];
    }

    // this block's keys are out before its ticket is
    __syncthreads();
    if (tid == 0) is_last = count_up(P.ticket, 1u, gridDim.x);
    __syncthreads();
    if (!is_last) return;

    // every key is final: accept lengths and tokens, as many sequences at a time as fit in shared memory (all
    // their keys in flight together); the keys go back to zero on the way, so that the scratch is ready for
    // the next call
    const int group = kGreedyTailRows / K1;
    for (int b0 = 0; b0 < P.B; b0 += group) {
        const int nb = min(group, P.B - b0), rows = nb * K1;
        for (int r = tid; r < rows; r += kGreedyThreads) {
            unsigned long long* kr = P.keys + (size_t)b0 * K1 + r;
            const int am = greedy_index(__ldcg(kr));
            *kr = 0ull;
            am_sh[r] = am;
            if (P.argmax) P.argmax[(size_t)b0 * K1 + r] = am;
            const int bl = r / K1, i = r - bl * K1;
            x_sh[r] = i < P.k ? P.x[(size_t)(b0 + bl) * P.k + i] : -1;
        }
        __syncthreads();
        for (int bl = tid; bl < nb; bl += kGreedyThreads) {
            int n = 0;
            while (n < P.k && x_sh[bl * K1 + n] == am_sh[bl * K1 + n]) ++n;
            P.accept_len[b0 + bl] = n;
            x_sh[bl * K1 + P.k] = n;
        }
        __syncthreads();
        for (int r = tid; r < rows; r += kGreedyThreads) {
            const int bl = r / K1, i = r - bl * K1, n = x_sh[bl * K1 + P.k];
            P.tokens[(size_t)b0 * K1 + r] = i <= n ? am_sh[r] : -1;      // accepted draft token = the argmax
        }
        __syncthreads();
    }
    if (tid == 0) *P.ticket = 0;   // leave the word ready for the next call
}

}  // namespace sdv
