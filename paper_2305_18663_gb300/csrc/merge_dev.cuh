// merge_dev.cuh -- device pieces of the block-merge proposals and their
// Delta DL (Alg. 1, Alg. 4), shared by the per-graph kernel (merge.cu) and
// the batched phase kernel (batch.cu), so that both score every proposal
// with the same arithmetic.
//
// Proposal i of block r (Philox counter (round_id, r, i), key (seed, 1)): u
// is the block at the far end of a uniformly chosen edge of block r (row r
// then column r of M); s != r is drawn with probability proportional to
// 1 + M[u][s] + M[s][u] (a uniform part over the other B-1 blocks, then row
// u and column u with block r left out).  A block with no edges draws s
// uniformly.
//
// Delta DL of merging r into s over rows and columns r, s only: row r moves
// into row s, column r into column s, the 2x2 corner collapses into M[s][s],
// and the block degrees of s absorb those of r.  Every term is
// f(a+b) - f(a) - f(b), f(x) = x ln x at integer counts, summed exactly in
// 128-bit fixed point from the table (FP64 a log1p(b/a) + b log1p(a/b) for
// counts beyond it), so the sum does not depend on its order and a block's
// entries can be spread over lanes and warps freely.  The model term of
// Eq. 2 is the same for every candidate and is left out.  The best proposal
// is the smallest score on a 2^-20-nat grid, earliest i on a tie.
//
// Work split.  A team of 1..8 warps takes a block.  Its lanes draw up to 32
// proposals at once (lane i draws proposal i with its corner and degree
// terms); then lane (g, q) sums the entries g, g + G, ... of row and column
// r for proposal q (G = 32 / proposals), so that an entry is read once for
// all proposals, every lookup is independent of the others, and four are in
// flight per lane.  Nonzero entries go through a small queue in shared
// memory, so that a dense row's zeros cost no lookups.
// Before, one warp walked the row once per proposal with FP64 log1p terms
// (1/64 rate: a term of 2 log1p and 2 divisions took some 1500 cycles of the
// SM).  Merge proposals of a 200k-vertex, 4M-edge graph, x = 10, before and
// after: B = 200,000 9.0 -> 2.2 ms, 25,000 10.4 -> 1.8 ms (sparse), 3125 dense
// 41.4 -> 0.39 ms, 1000 5.7 -> 0.14 ms.  What bounds it now is the latency of
// the dependent lookups (row offset, table slot, term).
#pragma once

#include <climits>
#include <cmath>

#include "common.cuh"

namespace sbp {
namespace {

constexpr int kMergeQueue = 160;  // entries queued per warp (worked off from 32 on, up to 128 join at a time)

// Proposal of block r on one lane (every search a single-lane one, so the
// lanes of a warp can draw different proposals of r at once).
template <bool SPARSE>
__device__ __forceinline__ int merge_propose(const ModelDev &md, int r, uint64_t w0, uint64_t w1) {
    const int B = md.B;
    const int64_t dr = (int64_t)md.dout[r] + md.din[r];
    if (dr == 0) {
        const int64_t y = draw_below(w1, (uint64_t)(B - 1));
        return (int)(y + (y >= r));
    }
    const int64_t t0 = draw_below(w0, (uint64_t)dr);
    int u;
    if (SPARSE) {
        u = sparse_cdf_block(md, r, (uint32_t)t0, (uint32_t)md.dout[r]);
    } else {
        u = (int)pivot_upper(md.P + (size_t)r * 2 * B, md.Pc + (size_t)r * 32, 0, 2 * B, (uint32_t)t0);
        if (u >= B) u -= B;
    }
    const int64_t Mur = Mat(md, u, r), Mru = Mat(md, r, u);
    const int64_t du_out = md.dout[u], du = du_out + md.din[u];
    const int64_t W = (B - 1) + du - Mur - Mru;
    const int64_t y = draw_below(w1, (uint64_t)W);
    if (y < B - 1) return (int)(y + (y >= r));
    const int64_t t = y - (B - 1);
    const int64_t row_w = du_out - Mur;
    if (SPARSE) {
        // the same walk over the nonzeros of row u or column u, entry r left
        // out (where it is zero there is nothing to step over)
        const bool row = t < row_w;
        const uint32_t a = (row ? md.rp : md.cp)[u], z = (row ? md.re : md.ce)[u];
        const uint32_t *prefix = row ? md.rpre : md.cpre;
        const int64_t own = row ? Mur : Mru;
        int64_t tt = row ? t : t - row_w;
        if (own != 0) {
            const uint32_t pos = lane_lower_i32(row ? md.rc : md.cr, a, z, r);
            const int64_t pre = pos > a ? (int64_t)prefix[pos - 1] : 0;
            if (tt >= pre) tt += own;
        }
        return (row ? md.rc : md.cr)[pivot_upper(prefix, (row ? md.rpc : md.cpc) + (size_t)u * 32, a, z, (uint32_t)tt)];
    }
    // dense: row u with column r left out, then column u with row r left out;
    // Pu[B + c] = dout_u + column prefix
    const uint32_t *Pu = md.P + (size_t)u * 2 * B;
    const bool row = t < row_w;
    const int64_t pre = row ? (r > 0 ? (int64_t)Pu[r - 1] : 0) : (r > 0 ? (int64_t)Pu[B + r - 1] : du_out);
    int64_t target = row ? t : du_out + (t - row_w);
    if (target >= pre) target += row ? Mur : Mru;
    return (int)pivot_upper(Pu, md.Pc + (size_t)u * 32, 0, 2 * B, (uint32_t)target) - (row ? 0 : B);
}

// a sum of terms: exact inside the table, FP64 beyond it
struct MergeSum {
    __int128 fix = 0;
    double fb = 0.0;
};

// adds (sub: takes away) f(a + b) - f(a) - f(b)
__device__ __forceinline__ void merge_term(const ModelDev &md, int64_t a, int64_t b, bool sub, MergeSum &s) {
    if (a == 0 || b == 0) return;
    if (a + b < md.XT) {
        const __int128 d = md.T[a + b] - md.T[a] - md.T[b];
        s.fix += sub ? -d : d;
    } else {
        const double d = gmerge(a, b);
        s.fb += sub ? -d : d;
    }
}

// The terms of merging r into s that do not come from row or column r's
// other entries, on one lane: the 2x2 corner collapsing into M[s][s]
// (added) and the block degrees of s absorbing those of r (subtracted).
__device__ __forceinline__ void merge_corner(const ModelDev &md, int r, int s, MergeSum &sum) {
    int Mrr, Mss, Mrs, Msr;
    Mat4corner(md, r, s, Mrr, Mss, Mrs, Msr);
    const int64_t a = Mrr, b = Mrs, c = Msr, d = Mss;
    merge_term(md, a, b, false, sum);
    merge_term(md, a + b, c, false, sum);
    merge_term(md, a + b + c, d, false, sum);
    merge_term(md, md.dout[s], md.dout[r], true, sum);
    merge_term(md, md.din[s], md.din[r], true, sum);
}

__device__ __forceinline__ long long score_key(double d) { return (long long)floor(d * 1048576.0 + 0.5); }

// the lane's place among the proposals: it sums for proposal q, which is s
// (row table of s at off, cap when sparse), the entries g, g + G, ...
struct MergeLane {
    int g, G, s;
    bool on;
    uint32_t off, cap;
};

// n queued entries (t, count; bit 31 of t set for a column entry M[t][r])
// against the lane's proposal
template <bool SPARSE>
__device__ __forceinline__ void merge_entries(const ModelDev &md, const int2 *queue, int n, const MergeLane &L,
                                              MergeSum &sum) {
    constexpr int kU = 4;
    for (int i0 = L.g; i0 < n; i0 += kU * L.G) {
        int a[kU], v[kU];
        if (SPARSE) {
            uint32_t off[kU], cap[kU], h[kU];
            int key[kU];
            int2 kv[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int i = i0 + u * L.G;
                const bool ok = L.on && i < n;
                const int2 e = ok ? queue[i] : make_int2(0, 0);
                const bool col = e.x < 0;
                const int t = e.x & 0x7fffffff;
                v[u] = (ok && t != L.s) ? e.y : 0;
                off[u] = L.off;
                cap[u] = L.cap;
                key[u] = t;
                if (v[u] != 0 && col) {
                    off[u] = md.hoff[t];
                    cap[u] = md.hoff[t + 1] - off[u];
                    key[u] = L.s;
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                h[u] = sparse_hash(key[u]) & (cap[u] - 1);
                kv[u] = v[u] != 0 ? md.hkv[off[u] + h[u]] : make_int2(-1, 0);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                a[u] = v[u] != 0 ? sparse_probe_from(md, off[u], cap[u], h[u], key[u], kv[u]) : 0;
        } else {
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int i = i0 + u * L.G;
                const bool ok = L.on && i < n;
                const int2 e = ok ? queue[i] : make_int2(0, 0);
                const int t = e.x & 0x7fffffff;
                v[u] = (ok && t != L.s) ? e.y : 0;
                a[u] = v[u] != 0 ? (e.x < 0 ? md.M[(size_t)t * md.B + L.s] : md.M[(size_t)L.s * md.B + t]) : 0;
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) merge_term(md, a[u], v[u], false, sum);
    }
}

// Entries of row and column r other than M[r][r], part `part` of `parts`,
// against the lane's proposal: 128 at a time (zeros dropped) join the warp's
// queue, which is worked off from 32 on.  (One call of merge_entries: at
// every place that found entries, its unrolled lookups filled the
// instruction cache, 7.5 of 21 cycles between two issues.)
template <bool SPARSE>
__device__ __forceinline__ void merge_rows(const ModelDev &md, int r, int part, int parts, int2 *queue,
                                           const MergeLane &L, MergeSum &sum) {
    const int lane = threadIdx.x & 31;
    uint32_t r0 = 0, c0 = 0, rlen = 0, total = (uint32_t)md.B;
    const int32_t *row = nullptr;
    const uint32_t *pre = nullptr;
    if (SPARSE) {
        r0 = md.rp[r];
        rlen = md.re[r] - r0;
        c0 = md.cp[r] - rlen;  // the column follows the row
        total = rlen + (md.ce[r] - md.cp[r]);
    } else {
        // the column's counts as differences of its prefix in P (coalesced;
        // pre[-1] is the end of the row's prefix, dout_r)
        row = md.M + (size_t)r * md.B;
        pre = md.P + (size_t)r * 2 * md.B + md.B;
    }
    int nq = 0;
    // the team's warps take chunks of 32 in turn, four (dense: two of the row
    // and two of the column) in flight
    const uint32_t next = 32u * parts, step = next * (SPARSE ? 4 : 2);
    for (uint32_t b0 = 32u * part;; b0 += step) {
        int2 e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int t, v = 0;
            if (SPARSE) {
                const uint32_t i = b0 + next * u + lane;
                const bool col = i >= rlen;
                t = i < total ? (col ? md.cr[c0 + i] : md.rc[r0 + i]) : r;
                if (t != r) v = col ? md.cv[c0 + i] : md.rv[r0 + i];
                t |= col ? INT32_MIN : 0;
            } else {
                t = (int)(b0 + next * (u >> 1) + lane);
                if (t < md.B && t != r) v = (u & 1) ? (int)(pre[t] - pre[t - 1]) : row[t];
                t |= (u & 1) ? INT32_MIN : 0;
            }
            e[u] = make_int2(t, v);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned nz = __ballot_sync(0xffffffffu, e[u].y != 0);
            if (e[u].y != 0) queue[nq + __popc(nz & ((1u << lane) - 1u))] = e[u];
            nq += __popc(nz);
        }
        const bool last = b0 >= total || total - b0 <= step;
        if (nq >= 32 || last) {
            __syncwarp();
            merge_entries<SPARSE>(md, queue, nq, L, sum);
            __syncwarp();
            nq = 0;
        }
        if (last) break;
    }
}

// the sums of the lanes (g, q) over g, on the lanes q of group 0
__device__ __forceinline__ void merge_fold(int nq, int G, MergeSum &sum) {
    const int lane = threadIdx.x & 31;
    const unsigned long long lo = (unsigned long long)sum.fix;
    const long long hi = (long long)(sum.fix >> 64);
    const double fb = sum.fb;
    for (int g = 1; g < G; ++g) {
        const int from = (lane + g * nq) & 31;
        const unsigned long long l2 = __shfl_sync(0xffffffffu, lo, from);
        const long long h2 = __shfl_sync(0xffffffffu, hi, from);
        sum.fix += (__int128)(((unsigned __int128)(unsigned long long)h2 << 64) | l2);
        sum.fb += __shfl_sync(0xffffffffu, fb, from);
    }
}

// Best proposal of block r by a team of `parts` warps (this one is number
// `part`).  team_sum(sum) adds the other warps' sums on lane q of warp 0 (a
// no-op for one warp); every warp of the team calls it the same number of
// times.  The result is valid in warp 0 (bs = -1 when x = 0).
template <bool SPARSE, class TeamSum>
__device__ __forceinline__ void merge_best(const ModelDev &md, uint64_t seed, uint64_t round_id, int x, int r,
                                           int part, int parts, int2 *queue, TeamSum team_sum, int &bs_out,
                                           double &bd_out) {
    const int lane = threadIdx.x & 31;
    int bs = -1;
    double bd = 0.0;
    long long bk = 0;
    for (int i0 = 0; i0 < x; i0 += 32) {
        const int nq = x - i0 < 32 ? x - i0 : 32;
        int si = 0;
        MergeSum corner;
        if (lane < nq) {
            const U64x4 w = philox4x64_10(round_id, (uint64_t)r, (uint64_t)(i0 + lane), 0, seed, 1);
            si = merge_propose<SPARSE>(md, r, w.x, w.y);
            if (part == 0) merge_corner(md, r, si, corner);
        }
        MergeLane L;
        L.G = 32 / nq;
        L.g = lane / nq;
        L.on = L.g < L.G;
        L.s = __shfl_sync(0xffffffffu, si, lane - L.g * nq);
        L.off = L.cap = 0;
        if (SPARSE) {
            L.off = md.hoff[L.s];
            L.cap = md.hoff[L.s + 1] - L.off;
        }
        MergeSum sum;
        merge_rows<SPARSE>(md, r, part, parts, queue, L, sum);
        merge_fold(nq, L.G, sum);
        sum.fix += corner.fix;
        sum.fb += corner.fb;
        team_sum(sum);
        const double d = -(fix_to_double(sum.fix) + sum.fb);
        // smallest score, then the earliest proposal
        const long long key = lane < nq ? score_key(d) : LLONG_MAX;
        long long kmin = key;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long k2 = __shfl_xor_sync(0xffffffffu, kmin, o);
            kmin = k2 < kmin ? k2 : kmin;
        }
        const int win = __ffs(__ballot_sync(0xffffffffu, lane < nq && key == kmin)) - 1;
        const int ws = __shfl_sync(0xffffffffu, si, win);
        const double wd = __shfl_sync(0xffffffffu, d, win);
        if (bs < 0 || kmin < bk) {
            bs = ws;
            bd = wd;
            bk = kmin;
        }
    }
    bs_out = bs;
    bd_out = bd;
}

}  // namespace
}  // namespace sbp
