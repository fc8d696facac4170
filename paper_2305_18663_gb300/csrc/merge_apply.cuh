// merge_apply.cuh -- the merge application of Alg. 1 ("sort best_merges",
// "pop, merge c into c'", pointer-based, Section III-A (d)) in parallel, by
// one thread block or by the thread blocks of one cluster.
//
// The rule: links r -> best_s[r] are taken in ascending (score on the
// 2^-20-nat grid, r); one is made unless its ends are in one group already;
// the rule stops at `want` links; groups are numbered by their smallest
// member.  Taking links in order and leaving out those that close a cycle is
// Kruskal's rule for the minimum spanning forest.  Every block has one
// outgoing link, so a connected set of links holds exactly one cycle (of two
// or more blocks), and the forest leaves out exactly that cycle's last link
// in the order.  So, without the sequential union-find:
//   1. pointer doubling finds the nodes on cycles (where paths of B or more
//      steps end) and every cycle's last link (the running maximum along the
//      doubled path); these links are rejected;
//   2. of the others, the `want` first in the order are made (a radix select
//      on the score's bits, ties by block id); a link among them is made
//      whatever comes after it, since rejection depends on earlier links
//      only;
//   3. the links made form a forest of pointers: pointer jumping gives the
//      roots, an atomic minimum the smallest members, a scan the labels.
// All of it is integer work with one result.  It is bound by the latency of
// the passes' gathers: log2 B passes for 1, about as many for 3.  The host
// form (scores read back, std::sort, a sequential union, the map sent) took
// 12 ms at 200,000 blocks; this takes 0.72 ms.
#pragma once

#include "common.cuh"
#include "merge_dev.cuh"

namespace sbp {
namespace {

// Work arrays of the application: B entries each; words of the team's scans
struct MergeApply {
    unsigned long long *key;
    int32_t *a0, *a1, *x0, *x1, *mark;
};
constexpr size_t kMergeApplyBytes = 28;  // per block

// exclusive scan over the block's threads (a multiple of 32, at most 1024);
// sh: 33 words.  Ends with a barrier, so sh can be used again.
__device__ __forceinline__ uint32_t cta_scan(uint32_t v, uint32_t *sh, uint32_t &total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        const uint32_t t = lane < nw ? sh[lane] : 0u;
        uint32_t z = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, z, o);
            if (lane >= o) z += y;
        }
        sh[lane] = z - t;
        if (lane == 31) sh[32] = z;
    }
    __syncthreads();
    const uint32_t r = sh[w] + x - v;
    total = sh[32];
    __syncthreads();
    return r;
}

// Shared memory of a team's block
struct TeamShared {
    uint32_t scan[33];
    uint32_t hist[256];
    uint32_t bin, before;
};

// One thread block.
struct CtaTeam {
    TeamShared &sh;
    __device__ int rank() const { return 0; }
    __device__ int size() const { return 1; }
    __device__ void sync() { __syncthreads(); }
    // the sum over the blocks of the team of a value each block holds in all
    // its threads, and what the blocks before this one hold
    __device__ uint32_t across(uint32_t v, uint32_t &before) {
        before = 0;
        return v;
    }
    // hist[bin] summed over the team (this thread's bin, threads below 256)
    __device__ uint32_t across_bins(uint32_t v) { return v; }
};

// The thread blocks of one cluster; they exchange through `words` in global
// memory (2 * 8 + 2 * 8 * 256 words), in two sets used in turn: a set is
// written again only after the barrier of the other set's use, which every
// block reaches after it has read the first.
struct ClusterTeam {
    TeamShared &sh;
    uint32_t *words;
    int turn = 0, turn_bins = 0;
    __device__ int rank() const { return cluster_rank(); }
    __device__ int size() const { return cluster_size(); }
    __device__ void sync() { cluster_sync(); }
    __device__ uint32_t across(uint32_t v, uint32_t &before) {
        uint32_t *w = words + 8 * turn;
        turn ^= 1;
        if (threadIdx.x == 0) w[rank()] = v;
        sync();
        uint32_t total = 0;
        before = 0;
        for (int c = 0; c < size(); ++c) {
            const uint32_t x = __ldcg(&w[c]);
            if (c < rank()) before += x;
            total += x;
        }
        return total;
    }
    __device__ uint32_t across_bins(uint32_t v) {
        uint32_t *w = words + 16 + 8 * 256 * turn_bins;
        turn_bins ^= 1;
        if (threadIdx.x < 256) w[rank() * 256 + threadIdx.x] = v;
        sync();
        uint32_t total = 0;
        if (threadIdx.x < 256)
            for (int c = 0; c < size(); ++c) total += __ldcg(&w[c * 256 + threadIdx.x]);
        return total;
    }
};
constexpr size_t kClusterWords = 16 + 2 * 8 * 256;

// exclusive scan over the team's threads, in (block, thread) order
template <class Team>
__device__ __forceinline__ uint32_t team_scan(Team &t, uint32_t v, uint32_t &total) {
    uint32_t mine, before;
    const uint32_t ex = cta_scan(v, t.sh.scan, mine);
    total = t.across(mine, before);
    return before + ex;
}

// later of two links in the order (score, block); -1 is none
__device__ __forceinline__ int later_link(const unsigned long long *key, int i, int j) {
    const unsigned long long a = key[i < 0 ? 0 : i], b = key[j < 0 ? 0 : j];
    const bool first = a > b || (a == b && i > j);
    return i < 0 ? j : j < 0 || first ? i : j;
}

// Makes the links and writes map[c], the new label of block c; returns the
// links made, B_new the new block count (the same on every thread of the
// team).  The team has at least 256 threads a block.
template <class Team>
__device__ int merge_apply(Team &tm, const MergeApply &W, int B, const int32_t *best_s, const double *best_d, int want,
                           int32_t *map, int &B_new) {
    const int nt = tm.size() * blockDim.x, tid = tm.rank() * blockDim.x + threadIdx.x;
    for (int r = tid; r < B; r += nt) {
        const int s = best_s[r];
        W.key[r] = (unsigned long long)score_key(best_d[r]) ^ 0x8000000000000000ull;  // unsigned order
        W.a0[r] = s >= 0 ? s : r;
        W.x0[r] = s >= 0 ? r : -1;
        W.mark[r] = 0;
    }
    tm.sync();
    // 1. where paths of 2^k >= B steps end, and their last links
    int32_t *a = W.a0, *an = W.a1, *x = W.x0, *xn = W.x1;
    for (int64_t len = 1; len < B; len <<= 1) {
        // four nodes' gathers in flight per thread
        for (int r0 = tid; r0 < B; r0 += 4 * nt) {
            int p[4], ap[4], xr[4], xp[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = r0 + u * nt;
                p[u] = r < B ? a[r] : 0;
                xr[u] = r < B ? x[r] : -1;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                ap[u] = a[p[u]];
                xp[u] = x[p[u]];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) xr[u] = later_link(W.key, xr[u], xp[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = r0 + u * nt;
                if (r < B) {
                    an[r] = ap[u];
                    xn[r] = xr[u];
                }
            }
        }
        tm.sync();
        int32_t *q = a;
        a = an;
        an = q;
        q = x;
        x = xn;
        xn = q;
    }
    for (int r = tid; r < B; r += nt) W.mark[a[r]] = 1;
    tm.sync();
    // the links that can be made (mark: 1), and the bits their scores differ in
    uint32_t n_can = 0;
    unsigned long long diff = 0;
    const unsigned long long key0 = W.key[0];
    for (int r = tid; r < B; r += nt) {
        const bool can = best_s[r] >= 0 && !(W.mark[r] && x[r] == r);
        W.mark[r] = can;
        n_can += can;
        diff |= W.key[r] ^ key0;
    }
    uint32_t total, unused;
    team_scan(tm, n_can, total);
    const int done = total < (uint32_t)want ? (int)total : want;
    // 2. the score of the last link made, and how many links of that score
    unsigned long long thr = ~0ull;
    uint32_t need = total;
    if (done < (int)total) {
        const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)diff);
        const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(diff >> 32));
        // the highest differing bit, as a count per byte boundary: the bytes
        // from the highest differing one down are walked
        const int mine = hi ? 64 - __clz((int)hi) : lo ? 32 - __clz((int)lo) : 0;
        if (threadIdx.x == 0) tm.sh.bin = 0;
        __syncthreads();
        if ((threadIdx.x & 31) == 0) atomicMax(&tm.sh.bin, (uint32_t)mine);
        __syncthreads();
        // (blocks agree on it through the histogram pass below: a maximum
        // over the team is the highest bit set in the sum of one-hot words)
        uint32_t hot = 0;
        const uint32_t top_bin = tm.sh.bin;
        __syncthreads();
        hot = tm.across_bins(threadIdx.x == top_bin ? 1u : 0u);
        if (threadIdx.x == 0) tm.sh.bin = 0;
        __syncthreads();
        if (hot) atomicMax(&tm.sh.bin, (uint32_t)threadIdx.x);
        __syncthreads();
        const int top = (int)tm.sh.bin;
        int shift = (top + 7) / 8 * 8;
        unsigned long long pref = shift >= 64 ? 0ull : key0 >> shift;
        need = (uint32_t)done;
        while (shift > 0) {
            if (threadIdx.x < 256) tm.sh.hist[threadIdx.x] = 0;
            __syncthreads();
            for (int r = tid; r < B; r += nt) {
                const unsigned long long k = W.key[r];
                if (W.mark[r] && (shift >= 64 || (k >> shift) == pref)) atomicAdd(&tm.sh.hist[(k >> (shift - 8)) & 255], 1u);
            }
            __syncthreads();
            const uint32_t c = tm.across_bins(threadIdx.x < 256 ? tm.sh.hist[threadIdx.x] : 0u);
            uint32_t all;
            const uint32_t ex = cta_scan(c, tm.sh.scan, all);
            if (ex < need && need <= ex + c) {
                tm.sh.bin = threadIdx.x;
                tm.sh.before = ex;
            }
            __syncthreads();
            pref = (pref << 8) | tm.sh.bin;
            need -= tm.sh.before;
            shift -= 8;
            __syncthreads();
        }
        thr = pref;
    }
    // the links made: scores below thr, and the first `need` blocks of score thr
    const int per = (B + nt - 1) / nt;
    const int lo_r = (int)((int64_t)tid * per < B ? (int64_t)tid * per : B);
    const int hi_r = lo_r + per < B ? lo_r + per : B;
    uint32_t eq = 0;
    for (int r = lo_r; r < hi_r; ++r) eq += W.mark[r] && W.key[r] == thr;
    uint32_t rank = team_scan(tm, eq, unused);
    for (int r = lo_r; r < hi_r; ++r) {
        bool take = W.mark[r] && W.key[r] < thr;
        if (W.mark[r] && W.key[r] == thr) take = rank++ < need;
        W.a0[r] = take ? best_s[r] : r;
    }
    tm.sync();
    // 3. roots by pointer jumping
    a = W.a0;
    an = W.a1;
    for (;;) {
        uint32_t changed = 0;
        for (int r = tid; r < B; r += nt) {
            const int p = a[r], q = a[p];
            an[r] = q;
            changed |= p != q;
        }
        int32_t *q = a;
        a = an;
        an = q;
        const uint32_t any = __syncthreads_or((int)changed) ? 1u : 0u;
        if (tm.across(any, unused) == 0) break;
    }
    // groups by their smallest member
    for (int r = tid; r < B; r += nt) W.x0[r] = B;
    tm.sync();
    for (int r = tid; r < B; r += nt) atomicMin(&W.x0[a[r]], r);
    tm.sync();
    uint32_t heads = 0;
    for (int r = lo_r; r < hi_r; ++r) heads += W.x0[a[r]] == r;
    uint32_t label = team_scan(tm, heads, total);
    for (int r = lo_r; r < hi_r; ++r)
        if (W.x0[a[r]] == r) W.x1[r] = (int32_t)label++;
    tm.sync();
    for (int r = tid; r < B; r += nt) map[r] = W.x1[W.x0[a[r]]];
    tm.sync();
    B_new = (int)total;
    return done;
}

// map[c]: the rank of c among the blocks that hold a vertex (present[c] > 0);
// returns their number
template <class Team>
__device__ int compact_map(Team &tm, int B, const int32_t *present, int32_t *map) {
    const int nt = tm.size() * blockDim.x, tid = tm.rank() * blockDim.x + threadIdx.x;
    const int per = (B + nt - 1) / nt;
    const int lo = (int)((int64_t)tid * per < B ? (int64_t)tid * per : B), hi = lo + per < B ? lo + per : B;
    uint32_t mine = 0, total;
    for (int c = lo; c < hi; ++c) mine += present[c] > 0;
    uint32_t label = team_scan(tm, mine, total);
    for (int c = lo; c < hi; ++c) map[c] = present[c] > 0 ? (int32_t)label++ : -1;
    tm.sync();
    return (int)total;
}

}  // namespace
}  // namespace sbp
