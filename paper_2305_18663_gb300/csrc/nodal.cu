// nodal.cu -- the asynchronous-Gibbs nodal decision pass of one graph.
//
// Vertices are split by total degree into three groups (k <= 32, 33..128,
// above 128), each with its own evaluation kernel: k_eval_batch (32 movers
// per warp; for 33..128 with direct-mapped counts while B is small),
// k_eval_warp_direct (one warp per mover, direct-mapped counts) or, at
// larger B, k_eval_table (one warp per mover with a shared-memory table) and
// k_eval_cta (one CTA per mover, the largest rows).  A small pass over all
// vertices is one kernel, k_eval_small, a warp per mover.  In a pass over all
// vertices without a trace the first two kinds draw the proposals of their
// group's vertices themselves; otherwise k_propose (one lane per vertex)
// draws every proposal first and hands the moving ones (s != r) over in
// lists by group.  Only movers' rows are aggregated.  Moves the FP32 test
// cannot settle are decided after the pass by the exact evaluation
// (k_eval_cta in recheck mode).  The decision goes to the pending
// assignment; M is untouched until commit.  The steps and their numerics
// are described in nodal_dev.cuh.
#include <algorithm>
#include <cmath>

#include "nodal_dev.cuh"

// CTAs per SM the evaluation kernels are compiled for (register budget:
// 80 registers at 3, 64 at 4; the direct-mapped kernel for the largest rows
// fits 4 without spilling once the exact evaluation is a kernel of its own)
#ifndef SBP_DECIDE_MIN_BLOCKS
#define SBP_DECIDE_MIN_BLOCKS 3
#endif
#ifndef SBP_DIRECT_MIN_BLOCKS
#define SBP_DIRECT_MIN_BLOCKS 4
#endif
// 1: full-range passes draw the proposals inside the evaluation kernels;
// 0: always k_propose first (for comparison builds)
#ifndef SBP_FUSED_PROPOSALS
#define SBP_FUSED_PROPOSALS 1
#endif

namespace sbp {
namespace {

// Proposal of every vertex in [v_begin, v_end).  Proposals with s = r end
// here; the others are appended to the list of their degree group.
__global__ void __launch_bounds__(256) k_propose(DecideArgs a) {
    const ModelDev &md = a.md;
    const GraphDev &g = a.g;
    const int lane = threadIdx.x & 31;
    Counts c;
    unsigned long long medges = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = a.v_begin + (int64_t)blockIdx.x * blockDim.x; base < a.v_end; base += stride) {
        const int64_t vv = base + threadIdx.x;
        int bin = -1, s = 0, v = (int)vv;
        uint64_t w2 = 0;
        if (vv < a.v_end && !(a.skip && a.skip[v])) {
            const Proposal p = propose_vertex(g, md, a.seed, a.sweep_id, v);
            s = p.s;
            if (p.k == 0) {
                write_trace(a, v, p.r, 0, 0.0, 0.0);
            } else if (p.s == p.r) {
                c.proposed++;
                write_trace(a, v, p.r, 1, 0.0, 0.0);
            } else {
                bin = p.k <= kSmallDeg ? 0 : p.k <= kWarpDeg ? 1 : !a.split_top || p.k <= kMidDeg ? 2 : p.k <= kWideDeg ? 3 : 4;
                w2 = p.w2;
                medges += (unsigned long long)p.k;
            }
        }
#pragma unroll
        for (int bb = 0; bb < kRecheck; ++bb) {
            const unsigned msk = __ballot_sync(0xffffffffu, bin == bb);
            if (msk == 0) continue;
            const int leader = __ffs(msk) - 1;
            unsigned pos0 = 0;
            if (lane == leader) pos0 = atomicAdd(&a.mcount[bb], (unsigned)__popc(msk));
            pos0 = __shfl_sync(0xffffffffu, pos0, leader);
            if (bin == bb) {
                Mover mv;
                mv.v = v;
                mv.s = s;
                mv.w2 = w2;
                a.movers[a.mbase[bb] + pos0 + __popc(msk & ((1u << lane) - 1u))] = mv;
            }
        }
    }
    flush_counts_warp(md, c, medges);
}

// ---------------------------------------------------------------------------
// One warp per mover at large B (B > kDirectMaxB): the row's neighbour blocks
// are counted in a shared-memory hash table of `cap` slots, then the entries
// are evaluated.  Warp w of W takes the movers w, w + W, ... of list `bin`.
//
// On sparse rows most of what an entry needs of M is zero, and looking it up
// costs two dependent loads of scattered sectors per count, four counts per
// entry.  The counts of row r, row s, column r and column s are contiguous in
// the CSR and CSC, so a row or column that is not much longer than the
// mover's own entry list (kStreamRatio) is read through instead, each of its
// entries looked up in the shared-memory table:
//   - a hit is one changed cell of M: its term of Delta L and its share of the
//     Hastings sums are added on the spot (all linear in the cells);
//   - hits in row s and column s mark their slot; the entries left unmarked
//     have a zero count there and get f(k) - f(0) in the pass over the
//     entries.  (Every entry with edges out of v has its cell in row r, and
//     every one with edges into v in column r.)
//   - the corner entries are the hits on r and s themselves.
// Longer rows (a hub's block) are probed entry by entry as before.
// Bound by instruction issue and the latency of those loads (36% of the issue
// slots, 4% of DRAM bandwidth).  A decision pass of 200k vertices, 4M edges
// (30% of the labels redrawn), with the tables sized by degree class: 845 ->
// 507 us at B = 4096 dense, 1679 -> 1231 us at B = 65,536 sparse.  The line
// kStreamRatio, at B = 65,536 / 8192: rows never read through 1443 / 1104 us,
// up to 2 entries per entry of the mover 1231 / 1061, 4 1233 / 1226, 8 1314 /
// 1362.
constexpr int kStreamRatio = 2;

struct TableWarp {
    int *keys;             // [cap] block, with the two mark bits; -1 empty
    unsigned *cnt;         // [cap] ko | ki << 16 (degrees below 65536)
    unsigned short *list;  // [cap] slots in order of appearance
    int *corner;           // [4] M[r][r], M[s][s], M[r][s], M[s][r]
    int2 *queue;           // [kTableQueue] changed cells waiting for their terms
    int cap, cap_log2;
};
constexpr int kTableIn = 4;                      // 32-entry chunks in flight
constexpr int kTableQueue = 31 + 32 * kTableIn;  // (an entry pushes at most four, too)
constexpr int kMarkRow = 1 << 29, kMarkCol = 1 << 30;  // hit in row s / column s
constexpr int kKeyMask = (1 << 24) - 1;

// a key's slot, -1 when it is not in the table (marks ignored)
__device__ __forceinline__ int table_find(const TableWarp &W, int key) {
    unsigned h = hash_slot(key, W.cap_log2);
    for (int p = 0; p < W.cap; ++p) {
        const int x = W.keys[h];
        if (x < 0) return -1;
        if ((x & kKeyMask) == key) return (int)h;
        h = (h + 1) & (unsigned)(W.cap - 1);
    }
    return -1;
}

// v's row into the table: the number of entries (in `list`), the self-loops
__device__ __forceinline__ int table_row(const DecideArgs &a, const TableWarp &W, int v, int o0, int i0, int kout, int k,
                                         int &self) {
    const int lane = threadIdx.x & 31;
    const ModelDev &md = a.md;
    constexpr int kIn = kTableIn;
    int nl = 0;
    self = 0;
    bool full = false;
    for (int base = 0; base < k; base += 32 * kIn) {
        int nb[kIn], tb[kIn];
        bool sf[kIn];
#pragma unroll
        for (int c4 = 0; c4 < kIn; ++c4) {
            const int idx = base + c4 * 32 + lane;
            nb[c4] = idx < k ? nb_raw(a.g, md, o0, i0, kout, idx) : 0;
        }
#pragma unroll
        for (int c4 = 0; c4 < kIn; ++c4) {
            const int idx = base + c4 * 32 + lane;
            sf[c4] = false;
            tb[c4] = idx < k ? nb_block(md, nb[c4], v, sf[c4]) : -1;
        }
#pragma unroll
        for (int c4 = 0; c4 < kIn; ++c4) {
            if (base + c4 * 32 >= k) break;
            const int idx = base + c4 * 32 + lane;
            const bool is_out = idx < kout, is_self = idx < k && sf[c4];
            self += __popc(__ballot_sync(0xffffffffu, is_self && is_out));
            bool fresh = false;
            unsigned h = 0;
            if (tb[c4] >= 0 && !is_self) {
                h = hash_slot(tb[c4], W.cap_log2);
                bool done = false;
                for (int p = 0; p < W.cap; ++p) {
                    const int prev = atomicCAS(&W.keys[h], -1, tb[c4]);
                    if (prev == -1 || prev == tb[c4]) {
                        fresh = prev == -1;
                        done = true;
                        break;
                    }
                    h = (h + 1) & (unsigned)(W.cap - 1);
                }
                if (done) atomicAdd(&W.cnt[h], is_out ? 1u : 0x10000u);
                else full = true;
            }
            const unsigned fm = __ballot_sync(0xffffffffu, fresh);
            if (fresh) W.list[nl + __popc(fm & ((1u << lane) - 1u))] = (unsigned short)h;
            nl += __popc(fm);
        }
    }
    if (full) record_status(md.status, SBP_EHASHFULL);
    __syncwarp();
    return nl;
}

// the sums of a move's entries on one lane
struct MoveSums {
    __int128 dl = 0;
    double fb = 0.0;
    float dlf = 0.0f, am = 0.0f, pf = 0.0f, pb = 0.0f;
};

// Changed cells of a move wait in the warp's queue as (m, k) for their terms
// f(m + k) - f(m) (bit 31 of m: subtracted, for the block degrees), so that
// the terms are evaluated by full warps and by one copy of their code: inline
// at every place that finds a cell, lanes without one idled and the kernel
// stalled on instruction fetches (5 of 13 cycles between two issues).
__device__ __forceinline__ void queue_cell(const TableWarp &W, int &nq, bool has, int m, int k) {
    const unsigned hm = __ballot_sync(0xffffffffu, has);
    if (has) W.queue[nq + __popc(hm & ((1u << (threadIdx.x & 31)) - 1u))] = make_int2(m, k);
    nq += __popc(hm);
}

template <bool DL32>
__device__ __forceinline__ void drain_cells(const ModelDev &md, const TableWarp &W, int &nq, int keep, MoveSums &S) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    while (nq > keep) {
        const int take = nq < 32 ? nq : 32;
        const int2 e = lane < take ? W.queue[nq - take + lane] : make_int2(0, 0);
        nq -= take;
        const int m = e.x & 0x7fffffff;
        if (DL32) {
            const float d = dxlogx32(m, e.y, S.am);
            S.dlf += e.x < 0 ? -d : d;
        } else {
            double f2 = 0.0;
            const __int128 d = dT(md.T, md.XT, m, e.y, f2);
            S.dl += e.x < 0 ? -d : d;
            S.fb += e.x < 0 ? -f2 : f2;
        }
    }
    __syncwarp();
}

// the move of x (entries in the table, nl of them) on sparse rows
template <bool DL32>
__device__ __forceinline__ void table_move_sparse(const DecideArgs &a, const TableWarp &W, VertexCtx &x, int nl,
                                                  uint64_t w2, Counts &c) {
    const int lane = threadIdx.x & 31;
    const ModelDev &md = a.md;
    const int r = x.r, s = x.s;
    // segments: row r, row s, column r, column s
    const uint32_t r0 = md.rp[r], r1 = md.re[r], s0 = md.rp[s], s1 = md.re[s];
    const uint32_t cr0 = md.cp[r], cr1 = md.ce[r], cs0 = md.cp[s], cs1 = md.ce[s];
    const uint32_t most = (uint32_t)(kStreamRatio * nl + 32);
    const bool st_r = r1 - r0 <= most, st_s = s1 - s0 <= most, st_cr = cr1 - cr0 <= most, st_cs = cs1 - cs0 <= most;
    const uint32_t e0 = st_r ? r1 - r0 : 0u, e1 = e0 + (st_s ? s1 - s0 : 0u), e2 = e1 + (st_cr ? cr1 - cr0 : 0u),
                   e3 = e2 + (st_cs ? cs1 - cs0 : 0u);
    const int deg = (lane < 6 ? md.dout : md.din)[(lane & 1) ? s : r];  // lanes 4..7: the degrees
    if (lane < 4) W.corner[lane] = 0;
    __syncwarp();
    MoveSums S;
    int nq = 0;
    constexpr int kIn = kTableIn;
    for (uint32_t b0 = 0; b0 < e3; b0 += 32 * kIn) {
        int key[kIn], val[kIn];
#pragma unroll
        for (int u = 0; u < kIn; ++u) {
            const uint32_t i = b0 + 32 * u + lane;
            const bool col = i >= e1;
            const uint32_t p = i < e0 ? r0 + i : i < e1 ? s0 + (i - e0) : i < e2 ? cr0 + (i - e1) : cs0 + (i - e2);
            key[u] = i < e3 ? (col ? md.cr : md.rc)[p] : -1;
            val[u] = i < e3 ? (col ? md.cv : md.rv)[p] : 0;
        }
#pragma unroll
        for (int u = 0; u < kIn; ++u) {
            if (b0 + 32 * u >= e3) break;
            const uint32_t i = b0 + 32 * u + lane;
            const bool col = i >= e1, to = col ? i >= e2 : i >= e0;  // to: of s, which the edges reach
            if (key[u] == r || key[u] == s) {
                // from rows r and s (the columns hold the same four again)
                if (!col) W.corner[!to ? (key[u] == r ? 0 : 2) : (key[u] == r ? 3 : 1)] = val[u];
                key[u] = -1;
            }
            const int slot = key[u] >= 0 ? table_find(W, key[u]) : -1;
            int kk = 0;
            if (slot >= 0) {
                const unsigned cc = W.cnt[slot];
                const int ko = (int)(cc & 0xffffu), ki = (int)(cc >> 16);
                kk = col ? ki : ko;  // rows change by ko, columns by ki
                if (to) atomicOr(&W.keys[slot], col ? kMarkCol : kMarkRow);
                const float cw = (float)(ko + ki) * md.rcp32[key[u]];
                if (to) S.pf += cw * (float)val[u];
                else S.pb += cw * (float)(val[u] - kk);
            }
            queue_cell(W, nq, kk != 0, val[u], to ? kk : -kk);
        }
        drain_cells<DL32>(md, W, nq, 31, S);
    }
    __syncwarp();
    // the counts to r and to s, and the corner entries not read through
    {
        const int slot = lane < 2 ? table_find(W, lane == 0 ? r : s) : -1;
        const unsigned cc = slot >= 0 ? W.cnt[slot] : 0u;
        const unsigned cr = __shfl_sync(0xffffffffu, cc, 0), cs = __shfl_sync(0xffffffffu, cc, 1);
        x.ko_r = (int)(cr & 0xffffu);
        x.ki_r = (int)(cr >> 16);
        x.ko_s = (int)(cs & 0xffffu);
        x.ki_s = (int)(cs >> 16);
    }
    int val = deg;
    if (lane < 4) {
        const bool of_r = lane == 0 || lane == 2;  // Mrr, Mrs
        val = (of_r ? st_r : st_s) ? W.corner[lane] : sparse_at(md, of_r ? r : s, (lane == 0 || lane == 3) ? r : s);
    }
    // the entries: what the hits left (an entry with ko > 0 has a cell in row
    // r, one with ki > 0 in column r, so those are hits where they were read)
    const bool all_read = st_r && st_s && st_cr && st_cs;
    for (int e0i = 0; e0i < nl; e0i += 32) {
        const int e = e0i + lane;
        const int slot = e < nl ? W.list[e] : 0;
        const int key = e < nl ? W.keys[slot] : r, t = key & kKeyMask;
        const bool on = t != r && t != s;
        const unsigned cc = on ? W.cnt[slot] : 0u;
        const int ko = (int)(cc & 0xffffu), ki = (int)(cc >> 16);
        const float cw = on ? (float)(ko + ki) * md.rcp32[t] : 0.0f;
        int Mst = 0, Mts = 0;
        if (!all_read) {
            int Mrt = ko, Mtr = ki;
            if (on) {
                if (!st_r) Mrt = sparse_at(md, r, t);
                if (!st_s) Mst = sparse_at(md, s, t);
                if (!st_cr) Mtr = sparse_at(md, t, r);
                if (!st_cs) Mts = sparse_at(md, t, s);
            }
            S.pf += cw * (float)(Mts + Mst);
            S.pb += cw * (float)((Mtr - ki) + (Mrt - ko));
            queue_cell(W, nq, !st_r && ko, Mrt, -ko);
            queue_cell(W, nq, !st_cr && ki, Mtr, -ki);
        }
        S.pf += cw;
        S.pb += cw;
        queue_cell(W, nq, ko && (!st_s || !(key & kMarkRow)), Mst, ko);
        queue_cell(W, nq, ki && (!st_cs || !(key & kMarkCol)), Mts, ki);
        drain_cells<DL32>(md, W, nq, 31, S);
    }
    // corner and degrees
    const int cr = x.ko_r + x.ki_r, cs = x.ko_s + x.ki_s;
    const int kk = lane == 0   ? -(cr + x.self)
                   : lane == 1 ? cs + x.self
                   : lane == 2 ? x.ki_r - x.ko_s
                   : lane == 3 ? x.ko_r - x.ki_s
                   : lane == 4 ? -x.Kout
                   : lane == 5 ? x.Kout
                   : lane == 6 ? -x.Kin
                               : x.Kin;
    queue_cell(W, nq, lane < 8 && kk != 0, lane < 4 ? val : val | INT32_MIN, kk);
    drain_cells<DL32>(md, W, nq, 0, S);
    CornerVals cv;
    cv.Mrr = __shfl_sync(0xffffffffu, val, 0);
    cv.Mss = __shfl_sync(0xffffffffu, val, 1);
    cv.Mrs = __shfl_sync(0xffffffffu, val, 2);
    cv.Msr = __shfl_sync(0xffffffffu, val, 3);
    cv.dr = md.dsum[r];
    cv.ds = md.dsum[s];
    float pf = warp_sum_f(S.pf), pb = warp_sum_f(S.pb);
    corner_hastings_fast(x, cv, md.B, pf, pb);
    // additions on a lane: one per 32 cells of the queue and one per 32
    // entries read; at most e3 + 4 nl + 8 cells (bounds all the FP32 sums)
    const int adds = (int)e3 + 4 * nl + 64;
    int dec = -1;
    if (DL32) {
        const float dlf = warp_sum_f(S.dlf), am = warp_sum_f(S.am);
        if (!a.trace_on) dec = fast_decision_f(a.beta32, dlf, 0.0f, pf, pb, w2, max(x.k, adds), dl32_error(am, adds));
    } else {
        const __int128 dl = warp_sum_128(S.dl);
        const bool has_fb = __any_sync(0xffffffffu, __double_as_longlong(S.fb) != 0);
        const double fb = has_fb ? warp_sum(S.fb) : 0.0;
        if (!a.trace_on) dec = fast_decision(a.beta32, dl, has_fb, fb, pf, pb, w2, max(x.k, adds));
    }
    if (lane == 0) {
        if (dec >= 0) {
            if (dec) accept_move(md, x.v, s, x.k);
            count_result(c, dec != 0, false, x.k);
        } else {
            push_recheck(a, x.v, s, w2);
        }
    }
}

template <bool DL32, bool SPARSE>
__global__ void __launch_bounds__(kWarpsPerCta * 32, SBP_DECIDE_MIN_BLOCKS) k_eval_table(DecideArgs a, int bin, int cap,
                                                                                     int cap_log2) {
    extern __shared__ int dsm[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const ModelDev &md = a.md;
    const GraphDev &g = a.g;
    TableWarp W;
    W.cap = cap;
    W.cap_log2 = cap_log2;
    __shared__ int2 queue[kWarpsPerCta][SPARSE ? kTableQueue : 1];
    __shared__ int corner[kWarpsPerCta][4];
    W.keys = dsm + (size_t)wid * cap;
    W.cnt = reinterpret_cast<unsigned *>(dsm + (size_t)nwarps * cap) + (size_t)wid * cap;
    W.list = reinterpret_cast<unsigned short *>(dsm + (size_t)2 * nwarps * cap) + (size_t)wid * cap;
    W.corner = corner[wid];
    W.queue = queue[wid];
    for (int i = lane; i < cap; i += 32) {
        W.keys[i] = -1;
        W.cnt[i] = 0;
    }
    __syncwarp();

    const Mover *mlist = a.movers + a.mbase[bin];
    const int64_t count = *(volatile unsigned *)&a.mcount[bin];
    Counts c;
    const int64_t gw = (int64_t)blockIdx.x * nwarps + wid, nw = (int64_t)gridDim.x * nwarps;
    // 32 movers' records at a time, a lane each
    for (int64_t j0 = 0; gw + j0 * nw < count; j0 += 32) {
        const int64_t i = gw + (j0 + lane) * nw;
        int pv = 0, ps = 0, pr = 0, po = 0, pko = 0, pi = 0, pki = 0;
        uint64_t pw2 = 0;
        if (i < count) {
            const Mover mv = mlist[i];
            pv = mv.v;
            ps = mv.s;
            pw2 = mv.w2;
            pr = md.b[pv];
            po = g.op[pv];
            pko = g.op[pv + 1] - po;
            pi = g.ip[pv];
            pki = g.ip[pv + 1] - pi;
        }
        const int nq = __popc(__ballot_sync(0xffffffffu, i < count));
        for (int q = 0; q < nq; ++q) {
            VertexCtx x;
            x.v = __shfl_sync(0xffffffffu, pv, q);
            x.s = __shfl_sync(0xffffffffu, ps, q);
            x.r = __shfl_sync(0xffffffffu, pr, q);
            const int o0 = __shfl_sync(0xffffffffu, po, q), i0 = __shfl_sync(0xffffffffu, pi, q);
            x.Kout = __shfl_sync(0xffffffffu, pko, q);
            x.Kin = __shfl_sync(0xffffffffu, pki, q);
            const uint64_t w2 = __shfl_sync(0xffffffffu, pw2, q);
            x.k = x.Kout + x.Kin;
            const int D = table_row(a, W, x.v, o0, i0, x.Kout, x.k, x.self);
            if (lane == 0) c.entries += (unsigned)D;
            if constexpr (SPARSE) {
                table_move_sparse<DL32>(a, W, x, D, w2, c);
            } else {
                evaluate_warp<DL32, false>(a, md, x, w2, [&](auto &&f) {
                    for (int e = lane; e < D; e += 32) {
                        const int slot = W.list[e];
                        const unsigned cc = W.cnt[slot];
                        f(W.keys[slot], (int)(cc & 0xffffu), (int)(cc >> 16));
                    }
                }, c);
            }
            __syncwarp();
            for (int e = lane; e < D; e += 32) {
                const int slot = W.list[e];
                W.keys[slot] = -1;
                W.cnt[slot] = 0;
            }
            __syncwarp();
        }
    }
    if (lane == 0) flush_counts(md, c);
}

// ---------------------------------------------------------------------------
// One warp per mover with direct-mapped counts (B <= kDirectMaxB): the row's
// neighbour blocks go straight into a per-warp array of B counts (ko | ki <<
// 16) with shared-memory atomics, the first touch of a block (an atomic that
// returns 0) appends it to the warp's list.  No table probing and no warp
// match; eight 32-edge chunks in flight per round.  Degrees below 65536.
constexpr int kDirectChunks = 8;

// one mover (v, s, w2) on the whole warp, counts in cnt[B] (all zero on entry
// and on return), first touches in list
template <bool DL32, bool EXACT>
__device__ __forceinline__ void direct_mover(const DecideArgs &a, unsigned *cnt, int *list, int v, int s, uint64_t w2,
                                             Counts &c) {
    const int lane = threadIdx.x & 31;
    const ModelDev &md = a.md;
    const GraphDev &g = a.g;
    const int r = md.b[v];
    const int o0 = g.op[v], kout = g.op[v + 1] - o0;
    const int i0 = g.ip[v], kin = g.ip[v + 1] - i0;
    const int k = kout + kin;
    int nl = 0, self = 0;
    for (int base = 0; base < k; base += 32 * kDirectChunks) {
        int nb[kDirectChunks], tb[kDirectChunks];
#pragma unroll
        for (int c8 = 0; c8 < kDirectChunks; ++c8) {
            const int idx = base + c8 * 32 + lane;
            nb[c8] = idx < k ? nb_raw(g, md, o0, i0, kout, idx) : 0;
        }
        bool sf[kDirectChunks];
#pragma unroll
        for (int c8 = 0; c8 < kDirectChunks; ++c8) {
            const int idx = base + c8 * 32 + lane;
            sf[c8] = false;
            tb[c8] = idx < k ? nb_block(md, nb[c8], v, sf[c8]) : -1;
        }
#pragma unroll
        for (int c8 = 0; c8 < kDirectChunks; ++c8) {
            const int idx = base + c8 * 32 + lane;
            const bool is_out = idx < kout, is_self = idx < k && sf[c8];
            self += __popc(__ballot_sync(0xffffffffu, is_self && is_out));
            bool fresh = false;
            if (tb[c8] >= 0 && !is_self) fresh = atomicAdd(&cnt[tb[c8]], is_out ? 1u : 0x10000u) == 0u;
            const unsigned fm = __ballot_sync(0xffffffffu, fresh);
            if (fresh) list[nl + __popc(fm & ((1u << lane) - 1u))] = tb[c8];
            nl += __popc(fm);
        }
    }
    __syncwarp();
    VertexCtx x;
    x.v = v; x.r = r; x.s = s;
    x.Kout = kout; x.Kin = kin; x.self = self; x.k = k;
    const int D = nl;
    if (lane == 0) c.entries += (unsigned)D;
    evaluate_warp<DL32, EXACT>(a, md, x, w2, [&](auto &&f) {
        for (int e = lane; e < D; e += 32) {
            const int t = list[e];
            const unsigned cc = cnt[t];
            f(t, (int)(cc & 0xffffu), (int)(cc >> 16));
        }
    }, c);
    __syncwarp();
    for (int e = lane; e < D; e += 32) cnt[list[e]] = 0u;
    __syncwarp();
}

// The proposals of vertices w, w + W, w + 2 W, ... of `count` (vertex(i) is
// the i-th), drawn one per lane, and the evaluation of the movers among them,
// one after another, on warp w of W.  Returns the lane's sum of its movers'
// degrees.
template <bool DL32, bool EXACT, class Vertex>
__device__ __forceinline__ unsigned long long direct_vertices(const DecideArgs &a, unsigned *cnt, int *list, int64_t gw,
                                                              int64_t nw, int64_t count, Vertex vertex, Counts &c) {
    const int lane = threadIdx.x & 31;
    unsigned long long medges = 0;
    for (int64_t j0 = 0; gw + j0 * nw < count; j0 += 32) {
        const int64_t i = gw + (j0 + lane) * nw;
        bool mover = false;
        int pv = 0, ps = 0;
        uint64_t pw = 0;
        if (i < count) {
            pv = vertex(i);
            const Proposal p = propose_vertex(a.g, a.md, a.seed, a.sweep_id, pv);
            if (p.s == p.r) {
                c.proposed++;
            } else {
                mover = true;
                ps = p.s;
                pw = p.w2;
                medges += (unsigned long long)p.k;
            }
        }
        unsigned mask = __ballot_sync(0xffffffffu, mover);
        while (mask) {
            const int q = __ffs(mask) - 1;
            mask &= mask - 1u;
            const int v = __shfl_sync(0xffffffffu, pv, q), s = __shfl_sync(0xffffffffu, ps, q);
            const uint64_t w2 = __shfl_sync(0xffffffffu, pw, q);
            direct_mover<DL32, EXACT>(a, cnt, list, v, s, w2, c);
        }
    }
    return medges;
}

// One warp per mover with direct-mapped counts.  FUSED = false: the movers
// of list `bin`.  FUSED = true: the warps draw the proposals of the group's
// vertices themselves (the group is sorted by descending degree, so every
// warp gets a share of the largest rows).
template <bool DL32, bool FUSED>
__global__ void __launch_bounds__(kWarpsPerCta * 32, SBP_DIRECT_MIN_BLOCKS) k_eval_warp_direct(DecideArgs a, int bin,
                                                                                           int warp_words) {
    extern __shared__ unsigned dmw[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const ModelDev &md = a.md;
    const int B = md.B;
    unsigned *cnt = dmw + (size_t)wid * warp_words;
    int *list = reinterpret_cast<int *>(cnt + B);
    for (int i = lane; i < B; i += 32) cnt[i] = 0u;
    __syncwarp();
    Counts c;
    const int64_t gw = (int64_t)blockIdx.x * nwarps + wid, nw = (int64_t)gridDim.x * nwarps;
    if constexpr (!FUSED) {
        const Mover *mlist = a.movers + a.mbase[bin];
        const int64_t count = *(volatile unsigned *)&a.mcount[bin];
        for (int64_t q = gw; q < count; q += nw) {
            const Mover mv = mlist[q];
            direct_mover<DL32, false>(a, cnt, list, mv.v, mv.s, mv.w2, c);
        }
        if (lane == 0) flush_counts(md, c);
    } else {
        const int32_t *vl = a.vlist[bin];
        const unsigned long long medges = direct_vertices<DL32, false>(
            a, cnt, list, gw, nw, a.vcount[bin], [&](int64_t i) { return vl[i]; }, c);
        flush_counts_warp(md, c, medges);
    }
}

// ---------------------------------------------------------------------------
// A small graph's whole pass in one launch: a warp per mover for every
// degree, the moves the FP32 test cannot settle decided on the spot.  The
// batches of 32 movers a warp (below) give a small graph too few warps, each
// with a long serial aggregation: the three groups' kernels and the recheck
// launch took 80 us at 1000 vertices and 107 us at 20,000 (16 edges out of
// each), this takes 11 and 39 us (where the line lies: small_pass).  It is bound by the chain of dependent
// loads of a proposal and a move, a few of them per warp.
template <bool DL32>
__global__ void __launch_bounds__(kWarpsPerCta * 32, 2) k_eval_small(DecideArgs a, int warp_words) {
    extern __shared__ unsigned smw[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const int B = a.md.B;
    unsigned *cnt = smw + (size_t)wid * warp_words;
    int *list = reinterpret_cast<int *>(cnt + B);
    for (int i = lane; i < B; i += 32) cnt[i] = 0u;
    __syncwarp();
    Counts c;
    const int64_t gw = (int64_t)blockIdx.x * nwarps + wid, nw = (int64_t)gridDim.x * nwarps;
    // the largest rows first
    const int64_t n2 = a.vcount[2], n1 = a.vcount[1];
    const unsigned long long medges = direct_vertices<DL32, true>(
        a, cnt, list, gw, nw, n2 + n1 + a.vcount[0], [&](int64_t i) {
            return i < n2 ? a.vlist[2][i] : i < n2 + n1 ? a.vlist[1][i - n2] : a.vlist[0][i - n2 - n1];
        }, c);
    flush_counts_warp(a.md, c, medges);
}

// ---------------------------------------------------------------------------
// CTA per mover: at large B the movers of more than kWideDeg edges, degrees of
// 65,536 and more at any B, and the recheck

struct CtaScratch {
    __int128 dl[kBigThreads / 32];
    double fb[kBigThreads / 32], pf64[kBigThreads / 32], pb64[kBigThreads / 32];
    float pf[kBigThreads / 32], pb[kBigThreads / 32], dlf[kBigThreads / 32], am[kBigThreads / 32];
    __int128 dl_tot;
    double fb_tot;
    int rs[4];
    int nlist, self, ok, dec;
};

// gtab: NULL, or a global scratch of 2 cap words per CTA for tables that do
// not fit shared memory
template <bool DL32>
__global__ void __launch_bounds__(kBigThreads) k_eval_cta(DecideArgs a, int bin, int cap, int cap_log2,
                                                          unsigned long long *gtab) {
    extern __shared__ unsigned long long smem_u64[];
    // CTAs beyond the list's length have nothing to do (the recheck launch
    // is usually nearly empty)
    if ((int64_t)blockIdx.x >= (int64_t)(*(volatile unsigned *)&a.mcount[bin])) return;
    unsigned long long *cnt = gtab ? gtab + (size_t)blockIdx.x * 2 * (size_t)cap : smem_u64;
    int *keys = reinterpret_cast<int *>(cnt + cap);
    int *list = keys + cap;
    __shared__ CtaScratch sh;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarps = kBigThreads / 32;
    for (int i = tid; i < cap; i += blockDim.x) {
        keys[i] = -1;
        cnt[i] = 0;
    }
    if (tid == 0) {
        sh.nlist = 0;
        sh.self = 0;
        sh.ok = 1;
    }
    __syncthreads();

    const GraphDev &g = a.g;
    const ModelDev &md = a.md;
    const Mover *mlist = a.movers + a.mbase[bin];
    const int64_t count = *(volatile unsigned *)&a.mcount[bin];
    Counts c;
    for (int64_t i = blockIdx.x; i < count; i += gridDim.x) {
        const Mover mv = mlist[i];
        const int v = mv.v, s = mv.s;
        const int r = md.b[v];
        const int o0 = g.op[v], kout = g.op[v + 1] - o0;
        const int i0 = g.ip[v], kin = g.ip[v + 1] - i0;
        const int k = kout + kin;
        if (tid < 4) sh.rs[tid] = 0;
        for (int base = 0; base < k; base += blockDim.x) {
            const int idx = base + tid;
            const bool valid = idx < k, is_out = idx < kout;
            bool sfl = false;
            const int tb = valid ? nb_block(md, nb_raw(g, md, o0, i0, kout, idx), v, sfl) : -1;
            const bool is_self = valid && sfl;
            const int nself = __popc(__ballot_sync(0xffffffffu, is_self && is_out));
            if (lane == 0 && nself) atomicAdd(&sh.self, nself);
            const int key = (valid && !is_self) ? tb : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, key);
            const unsigned outm = __ballot_sync(0xffffffffu, valid && !is_self && is_out);
            if (key >= 0 && lane == __ffs(peers) - 1) {
                const unsigned ko = __popc(peers & outm), ki = __popc(peers) - ko;
                if (!table_add(keys, cnt, list, &sh.nlist, cap, cap_log2, key,
                               (unsigned long long)ko | ((unsigned long long)ki << 32)))
                    sh.ok = 0;
            }
        }
        __syncthreads();
        const int D = sh.nlist;
        if (tid == 0 && !sh.ok) record_status(md.status, SBP_EHASHFULL);
        if (tid == 0 && !a.force_exact) c.entries += (unsigned)D;
        VertexCtx x;
        x.v = v; x.r = r; x.s = s;
        x.Kout = kout; x.Kin = kin; x.self = sh.self; x.k = k;
        for (int e = tid; e < D; e += blockDim.x) {
            const int slot = list[e];
            const int t = keys[slot];
            const unsigned long long cc = cnt[slot];
            if (t == r) { sh.rs[0] = (int)(cc & 0xffffffffu); sh.rs[1] = (int)(cc >> 32); }
            if (t == s) { sh.rs[2] = (int)(cc & 0xffffffffu); sh.rs[3] = (int)(cc >> 32); }
        }
        __syncthreads();
        x.ko_r = sh.rs[0]; x.ki_r = sh.rs[1]; x.ko_s = sh.rs[2]; x.ki_s = sh.rs[3];
        __int128 dl = 0;
        double fb = 0.0;
        float pf = 0.0f, pb = 0.0f, dlf = 0.0f, am = 0.0f;
        // the FP32 pass only feeds the FP32 test; when the exact evaluation
        // decides anyway (the recheck launch, a trace) it is skipped (the
        // exact form's pass also yields the exact Delta L, so it stays)
        const bool fast_pass = !DL32 || (!a.trace_on && !a.force_exact);
        for (int e = tid; fast_pass && e < D; e += blockDim.x) {
            const int slot = list[e];
            const int t = keys[slot];
            const unsigned long long cc = cnt[slot];
            if (t != r && t != s) {
                if (DL32)
                    entry_fast32(md, x, t, (int)(cc & 0xffffffffu), (int)(cc >> 32), dlf, am, pf, pb);
                else
                    entry_fast(md, x, t, (int)(cc & 0xffffffffu), (int)(cc >> 32), dl, fb, pf, pb);
            }
        }
        if (fast_pass && tid < 32) {
            if (DL32)
                special_terms32(md, x, tid, dlf, am);
            else
                special_terms(md, x, tid, dl, fb);
        }
        pf = warp_sum_f(pf);
        pb = warp_sum_f(pb);
        if (DL32) {
            dlf = warp_sum_f(dlf);
            am = warp_sum_f(am);
        } else {
            dl = warp_sum_128(dl);
            if (__any_sync(0xffffffffu, __double_as_longlong(fb) != 0)) fb = warp_sum(fb);
        }
        if (lane == 0) {
            sh.dl[wid] = dl;
            sh.fb[wid] = fb;
            sh.pf[wid] = pf;
            sh.pb[wid] = pb;
            sh.dlf[wid] = dlf;
            sh.am[wid] = am;
        }
        __syncthreads();
        CornerVals cv;
        Mat4corner(md, r, s, cv.Mrr, cv.Mss, cv.Mrs, cv.Msr);
        cv.dr = md.dsum[r];
        cv.ds = md.dsum[s];
        if (tid == 0) {
            __int128 dlt = 0;
            double fbt = 0.0;
            float pft = 0.0f, pbt = 0.0f, dlft = 0.0f, amt = 0.0f;
            for (int q = 0; q < nwarps; ++q) {
                dlt += sh.dl[q];
                fbt += sh.fb[q];
                pft += sh.pf[q];
                pbt += sh.pb[q];
                dlft += sh.dlf[q];
                amt += sh.am[q];
            }
            sh.dl_tot = dlt;
            sh.fb_tot = fbt;
            corner_hastings_fast(x, cv, md.B, pft, pbt);
            int dec = -1;
            if (!a.trace_on && !a.force_exact) {
                if (DL32)
                    dec = fast_decision_f(a.beta32, dlft, 0.0f, pft, pbt, mv.w2, k, dl32_error(amt, k));
                else
                    dec = fast_decision(a.beta32, dlt, __double_as_longlong(fbt) != 0, fbt, pft, pbt, mv.w2, k);
            }
            sh.dec = dec;
            if (dec >= 0) {
                if (dec) accept_move(md, v, s, x.k);
                count_result(c, dec != 0, false, x.k);
            }
        }
        __syncthreads();
        if (sh.dec < 0) {
            double pf64 = 0.0, pb64 = 0.0;
            __int128 dle = 0;
            double fbe = 0.0;
            for (int e = tid; e < D; e += blockDim.x) {
                const int slot = list[e];
                const int t = keys[slot];
                const unsigned long long cc = cnt[slot];
                if (t != r && t != s) {
                    if (DL32)
                        entry_exact_all(md, x, t, (int)(cc & 0xffffffffu), (int)(cc >> 32), dle, fbe, pf64, pb64);
                    else
                        entry_exact(md, x, t, (int)(cc & 0xffffffffu), (int)(cc >> 32), pf64, pb64);
                }
            }
            if (DL32) {
                if (tid < 32) special_terms(md, x, tid, dle, fbe);
                dle = warp_sum_128(dle);
                if (__any_sync(0xffffffffu, __double_as_longlong(fbe) != 0)) fbe = warp_sum(fbe);
                if (lane == 0) {
                    sh.dl[wid] = dle;
                    sh.fb[wid] = fbe;
                }
            }
            pf64 = warp_sum(pf64);
            pb64 = warp_sum(pb64);
            if (lane == 0) {
                sh.pf64[wid] = pf64;
                sh.pb64[wid] = pb64;
            }
            __syncthreads();
            if (tid == 0) {
                double pft = 0.0, pbt = 0.0;
                __int128 dlt = sh.dl_tot;
                double fbt = sh.fb_tot;
                if (DL32) {
                    dlt = 0;
                    fbt = 0.0;
                    for (int q = 0; q < nwarps; ++q) {
                        dlt += sh.dl[q];
                        fbt += sh.fb[q];
                    }
                }
                for (int q = 0; q < nwarps; ++q) {
                    pft += sh.pf64[q];
                    pbt += sh.pb64[q];
                }
                corner_hastings_exact(x, cv, md.B, pft, pbt);
                const Exact e = exact_decision(a.beta, dlt, fbt, pft, pbt, mv.w2);
                if (e.accept) accept_move(md, v, s, k);
                count_exact(c, e.accept, e.margin, k);
                write_trace(a, v, s, 1 | (e.accept ? 2 : 0) | (e.margin ? 4 : 0), e.dH, e.logA);
            }
        }
        __syncthreads();
        for (int e = tid; e < D; e += blockDim.x) {
            const int slot = list[e];
            keys[slot] = -1;
            cnt[slot] = 0;
        }
        if (tid == 0) {
            sh.nlist = 0;
            sh.self = 0;
        }
        __syncthreads();
    }
    if (tid == 0) flush_counts(md, c);
}

// ---------------------------------------------------------------------------
// moves of vertices with 1 <= k <= 32: batches of 32 movers per warp
//
//   P1 lane per mover: record, offsets, label; exclusive prefix of k;
//   P2 edge parallel over the batch's concatenated rows (four 32-wide
//      chunks in flight): neighbour blocks into shared memory, tagged with
//      the mover's slot;
//   P3 windows of whole rows (at most 32 edge ends): match/ballot
//      aggregation into (q, t, kout, kin) entries, compacted in place, in
//      row order;
//   P5 entry parallel: Delta L (table sums, per entry in 64-bit fixed point
//      at 2^-48) and FP32 Hastings terms, summed per mover by a segmented
//      warp scan (entries of a mover are contiguous);
//   P6 lane per mover: corner and degree terms, FP32 test with its band;
//      a move the band does not settle goes to the recheck list.

// rows of at most 32 edges: sub-batches of 512 edge ends keep a CTA's
// shared memory at 38 KB, so that 4 CTAs (64 registers each) fit an SM
#ifndef SBP_BATCH0_EDGES
#define SBP_BATCH0_EDGES 512
#endif
#ifndef SBP_BATCH0_MIN_BLOCKS
#define SBP_BATCH0_MIN_BLOCKS 4
#endif
// CTAs of eight warps per SM (register budgets) of the batch kernels.  MANY:
// the FP32 form's budgets also for the exact form, whose 128-bit sums spill
// there.  Fewer warps without spills are the faster form in a pass of one or
// two waves, more warps in a long one over the first group (its lines are in
// launch_groups).
constexpr int batch_min_blocks(int mode, bool dl32, bool many) {
    const bool most = dl32 || many;
    return mode == 0 ? (most ? SBP_BATCH0_MIN_BLOCKS : 3) : (most ? SBP_DECIDE_MIN_BLOCKS : 2);
}
// edge ends per sub-batch (33..128).  Fewer (kBatchFewer) leave more shared
// memory to CTAs and to the L1 cache, which the long chains of the exact form
// and of sparse rows use; at few blocks there is room anyway, at many the
// counts take it all the same, and rows of 80 edges need more sub-batches.
// 1024 and 768 in us, B = 50 / 316 / 1000: 600,000 vertices of 40 edges, sparse
// 633 and 614 / 711 and 642 / 742 and 792; dense 594 and 581 / 620 and 587 /
// 677 and 687; of 80 edges, dense 843 and 883 / 919 and 951 / 1061 and 1098;
// 60,000 vertices of 67 edges, sparse 145 and 144 / 181 and 164 / 184 and 202.
constexpr int kBatchEdges = 1024, kBatchFewer = 768;
constexpr int kBatchEdges0 = SBP_BATCH0_EDGES;  // ... for rows of at most 32
constexpr int kDirectMaxB = 2048;  // direct-mapped per-warp counts up to this B

template <int EDGES>
struct BatchWarpT {
    int key[EDGES];  // edge ends (q << 26 | self << 25 | t << 1 | in), then entries (q << 26 | t)
    unsigned short ec[EDGES];  // entry counts ko | ki << 8
    int r[32], s[32], rsr[32], rss[32], hasfb[32];
    long long dl[32];  // Delta L, fixed point 2^-48
    float pf[32], pb[32];
    float dlf[32], am[32];  // FP32 Delta L and its magnitude sum (precision form)
    double fb[32];
};


__device__ __forceinline__ float fix48_to_float(long long v) {
    return fmaf((float)(int)(v >> 32), 0x1p-16f, (float)(unsigned)(v & 0xffffffffu) * 0x1p-48f);
}
__device__ __forceinline__ double fix48_to_double(long long v) {
    return (double)(int)(v >> 32) * 0x1p-16 + (double)(unsigned)(v & 0xffffffffu) * 0x1p-48;
}

// The evaluation of up to 32 movers of one warp: lane q < nv holds mover q
// (v, s, w2).  MODE 0: rows of at most 32 edges (aggregated in windows of
// whole rows); MODE 1: rows of 33..128 edges (aggregated per mover in a
// direct-mapped count array of B entries, dcnt, with its touch list dlist,
// which follow the warp's BatchWarp in shared memory).  Movers are taken in
// sub-batches of at most kEdges edge ends.
template <int MODE, bool DL32, int kEdges>
__device__ __forceinline__ void batch_movers(const DecideArgs &a, BatchWarpT<kEdges> &W, unsigned *dcnt, int *dlist,
                                             const int nv, int v, int s, uint64_t w2, Counts &c) {
    const int lane = threadIdx.x & 31;
    const GraphDev &g = a.g;
    const ModelDev &md = a.md;
    const int B = md.B;
    // ---- P1 (the mover records are in registers)
    int r = 0, o0 = 0, kout = 0, i0 = 0, kin = 0, k = 0;
    if (lane < nv) {
        r = md.b[v];
        o0 = g.op[v];
        kout = g.op[v + 1] - o0;
        i0 = g.ip[v];
        kin = g.ip[v + 1] - i0;
        k = kout + kin;
    } else {
        v = 0;
        s = -1;
        w2 = 0;
    }
    int incl = k;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int first = incl - k;
    // sub-batches of whole rows with at most kEdges edge ends
    for (int sa = 0; sa < nv;) {
    const int fs = __shfl_sync(0xffffffffu, first, sa);
    const unsigned fit = __ballot_sync(0xffffffffu, lane >= sa && lane < nv && incl - fs <= kEdges);
    const int sb = 31 - __clz(fit);
    const int total = __shfl_sync(0xffffffffu, incl, sb) - fs;
    const bool act = lane >= sa && lane <= sb;
    // ---- P2 (eight 32-edge chunks in flight for the longer rows of MODE 1)
    constexpr int kP2 = MODE == 1 ? 8 : 4;
    for (int base = 0; base < total; base += 32 * kP2) {
        int nb[kP2], vq[kP2], tag[kP2];
#pragma unroll
        for (int c4 = 0; c4 < kP2; ++c4) {
            const int pp = base + c4 * 32 + lane;
            const int p = fs + pp;
            int q = 0;
#pragma unroll
            for (int st = 16; st >= 1; st >>= 1) {
                const int f = __shfl_sync(0xffffffffu, first, q + st);
                if (f <= p) q += st;
            }
            const int fq = __shfl_sync(0xffffffffu, first, q);
            const int kq = __shfl_sync(0xffffffffu, kout, q);
            const int oq = __shfl_sync(0xffffffffu, o0, q);
            const int iq = __shfl_sync(0xffffffffu, i0, q);
            vq[c4] = __shfl_sync(0xffffffffu, v, q);
            const int e = p - fq;
            tag[c4] = (q << 26) | (e < kq ? 0 : 1);
            nb[c4] = pp < total ? nb_raw(g, md, oq, iq, kq, e) : 0;
        }
#pragma unroll
        for (int c4 = 0; c4 < kP2; ++c4) {
            const int pp = base + c4 * 32 + lane;
            if (pp < total) {
                bool sfl;
                const int t = nb_block(md, nb[c4], vq[c4], sfl);
                W.key[pp] = sfl ? (tag[c4] | (1 << 25)) : (tag[c4] | (t << 1));
            }
        }
    }
    __syncwarp();
    int nent = 0, my_self = 0, my_est = 0, my_ecnt = 0;
    if (MODE == 0) {
    // ---- P3: windows of whole rows
    for (int qa = sa; qa <= sb;) {
        const int fa = __shfl_sync(0xffffffffu, first, qa);
        const unsigned inw = __ballot_sync(0xffffffffu, lane >= qa && lane <= sb && incl - fa <= 32);
        const int qb = 31 - __clz(inw);
        const int wend = __shfl_sync(0xffffffffu, incl, qb);
        const int p = fa + lane;
        const bool valid = p < wend;
        const int x = valid ? W.key[p - fs] : 0;
        const bool selfl = valid && ((x >> 25) & 1);
        const bool in = (x & 1) != 0;
        const bool isent = valid && !selfl;
        const int mkey = isent ? (x >> 1) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, mkey);
        const unsigned outm = __ballot_sync(0xffffffffu, isent && !in);
        const unsigned sfl = __ballot_sync(0xffffffffu, selfl && !in);
        const bool leader = isent && lane == __ffs(peers) - 1;
        const unsigned lm = __ballot_sync(0xffffffffu, leader);
        if (leader) {
            const int ko = __popc(peers & outm), ki = __popc(peers) - ko;
            const int pos = nent + __popc(lm & ((1u << lane) - 1u));
            W.key[pos] = (x & (31 << 26)) | ((x >> 1) & 0xffffff);
            W.ec[pos] = (unsigned short)(ko | (ki << 8));
        }
        if (lane >= qa && lane <= qb) {
            const int lo_l = first - fa, hi_l = incl - fa;
            const unsigned below = (1u << lo_l) - 1u;
            const unsigned mq = (hi_l >= 32 ? 0xffffffffu : ((1u << hi_l) - 1u)) & ~below;
            my_self = __popc(sfl & mq);
            my_est = nent + __popc(lm & below);
            my_ecnt = __popc(lm & mq);
        }
        nent += __popc(lm);
        qa = qb + 1;
    }
    } else {
    // ---- P3: per mover, direct-mapped counts; first touches kept in
    // order of appearance (ballot compaction), so entries are deterministic
    for (int q = sa; q <= sb; ++q) {
        const int kq = __shfl_sync(0xffffffffu, k, q);
        const int fq = __shfl_sync(0xffffffffu, first, q) - fs;
        int nl = 0, selfq = 0;
        for (int c0 = 0; c0 < kq; c0 += 32) {
            const bool valid = c0 + lane < kq;
            const int x = valid ? W.key[fq + c0 + lane] : 0;
            const bool selfl = valid && ((x >> 25) & 1);
            const bool in = (x & 1) != 0;
            const bool isent = valid && !selfl;
            const int t = isent ? ((x >> 1) & 0xffffff) : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, t);
            const unsigned outm = __ballot_sync(0xffffffffu, isent && !in);
            selfq += __popc(__ballot_sync(0xffffffffu, selfl && !in));
            const bool leader = isent && lane == __ffs(peers) - 1;
            bool fresh = false;
            if (leader) {
                const unsigned ko = __popc(peers & outm), ki = __popc(peers) - ko;
                fresh = atomicAdd(&dcnt[t], ko | (ki << 16)) == 0u;
            }
            const unsigned fm = __ballot_sync(0xffffffffu, fresh);
            if (fresh) dlist[nl + __popc(fm & ((1u << lane) - 1u))] = t;
            nl += __popc(fm);
            __syncwarp();
        }
        for (int e = lane; e < nl; e += 32) {
            const int t = dlist[e];
            const unsigned cc = dcnt[t];
            dcnt[t] = 0u;
            W.key[nent + e] = (q << 26) | t;
            W.ec[nent + e] = (unsigned short)((cc & 0xffu) | ((cc >> 16) << 8));
        }
        if (lane == q) {
            my_self = selfq;
            my_est = nent;
            my_ecnt = nl;
        }
        nent += nl;
        __syncwarp();
    }
    }
    W.r[lane] = r;
    W.s[lane] = act ? s : -1;
    W.rsr[lane] = 0;
    W.rss[lane] = 0;
    W.hasfb[lane] = 0;
    W.dl[lane] = 0;
    W.pf[lane] = 0.0f;
    W.pb[lane] = 0.0f;
    W.dlf[lane] = 0.0f;
    W.am[lane] = 0.0f;
    W.fb[lane] = 0.0;
    __syncwarp();
    // ---- P5: entry parallel, segmented sums per mover
    for (int base = 0; base < nent; base += 32) {
        const int e = base + lane;
        const bool valid = e < nent;
        const unsigned ent = valid ? (unsigned)W.key[e] : 0u;
        const int q = valid ? (int)(ent >> 26) : 32;
        long long d48 = 0;
        float pfe = 0.0f, pbe = 0.0f, dlf = 0.0f, am = 0.0f;
        double f = 0.0;
        if (valid) {
            const int t = (int)(ent & 0x3ffffffu);
            const unsigned ec = W.ec[e];
            const int ko = (int)(ec & 0xffu), ki = (int)(ec >> 8);
            const int rq = W.r[q], sq = W.s[q];
            if (t == rq) {
                W.rsr[q] = ko | (ki << 8);
            } else if (t == sq) {
                W.rss[q] = ko | (ki << 8);
            } else {
                VertexCtx x;
                x.r = rq;
                x.s = sq;
                if (DL32) {
                    entry_fast32(md, x, t, ko, ki, dlf, am, pfe, pbe);
                } else {
                    __int128 d = 0;
                    entry_fast(md, x, t, ko, ki, d, f, pfe, pbe);
                    d48 = (long long)(d >> 16);
                }
            }
        }
        const bool anyfb = !DL32 && __any_sync(0xffffffffu, __double_as_longlong(f) != 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int qo = __shfl_up_sync(0xffffffffu, q, o);
            const float p2 = __shfl_up_sync(0xffffffffu, pfe, o);
            const float b2 = __shfl_up_sync(0xffffffffu, pbe, o);
            if (DL32) {
                const float l2 = __shfl_up_sync(0xffffffffu, dlf, o);
                const float a2 = __shfl_up_sync(0xffffffffu, am, o);
                if (lane >= o && qo == q) {
                    dlf += l2;
                    am += a2;
                }
            } else {
                const long long d2 = __shfl_up_sync(0xffffffffu, d48, o);
                if (lane >= o && qo == q) d48 += d2;
            }
            if (lane >= o && qo == q) {
                pfe += p2;
                pbe += b2;
            }
        }
        if (anyfb) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int qo = __shfl_up_sync(0xffffffffu, q, o);
                const double f2 = __shfl_up_sync(0xffffffffu, f, o);
                if (lane >= o && qo == q) f += f2;
            }
        }
        const int qn = __shfl_down_sync(0xffffffffu, q, 1);
        if (valid && (lane == 31 || qn != q)) {
            if (DL32) {
                W.dlf[q] += dlf;
                W.am[q] += am;
            } else {
                W.dl[q] += d48;
            }
            W.pf[q] += pfe;
            W.pb[q] += pbe;
            if (anyfb && __double_as_longlong(f) != 0) {
                W.fb[q] += f;
                W.hasfb[q] = 1;
            }
        }
        __syncwarp();
    }
    __syncwarp();
    // ---- P6: lane per mover
    if (act) {
        c.entries += (unsigned)my_ecnt;
        VertexCtx x;
        x.v = v; x.r = r; x.s = s;
        x.Kout = kout; x.Kin = kin; x.self = my_self; x.k = k;
        const int rsr = W.rsr[lane], rss = W.rss[lane];
        x.ko_r = rsr & 0xff; x.ki_r = rsr >> 8;
        x.ko_s = rss & 0xff; x.ki_s = rss >> 8;
        __int128 d = 0;
        bool has_fb = W.hasfb[lane] != 0;
        double fb = has_fb ? W.fb[lane] : 0.0;
        float dlf = W.dlf[lane], am = W.am[lane];
        CornerVals cv;
        if (DL32) {
            cv = special_terms32_lane(md, x, dlf, am);
        } else {
            cv.Mrr = special_terms(md, x, 0, d, fb);
            cv.Mss = special_terms(md, x, 1, d, fb);
            cv.Mrs = special_terms(md, x, 2, d, fb);
            cv.Msr = special_terms(md, x, 3, d, fb);
#pragma unroll
            for (int jj = 4; jj < 8; ++jj) special_terms(md, x, jj, d, fb);
            has_fb = has_fb || __double_as_longlong(fb) != 0;
        }
        cv.dr = md.dsum[r];
        cv.ds = md.dsum[s];
        long long dl48 = W.dl[lane] + (long long)(d >> 16);
        float pf = W.pf[lane], pb = W.pb[lane];
        corner_hastings_fast(x, cv, B, pf, pb);
        int dec = -1;
        if (!a.trace_on) {
            if (DL32)
                dec = fast_decision_f(a.beta32, dlf, 0.0f, pf, pb, w2, k, dl32_error(am, k));
            else
                dec = fast_decision_f(a.beta32, fix48_to_float(dl48), has_fb ? (float)fb : 0.0f, pf, pb, w2, k);
        }
        if (dec >= 0) {
            if (dec) accept_move(md, v, s, k);
            count_result(c, dec != 0, false, k);
        } else {
            push_recheck(a, v, s, w2);  // the exact evaluation follows the pass
        }
    }
    __syncwarp();
        sa = sb + 1;
    }
}

// k_eval_batch: 32 movers per warp.  FUSED = false: the movers come from the
// list of degree group `bin` that k_propose filled.  FUSED = true: the warps
// draw the proposals of that group's vertices themselves (32 per round, lane
// per vertex), keep the movers in a queue of two slots per lane (position p
// in lane p % 32, slot p / 32) and evaluate them 32 at a time, so that the
// proposals' load chains overlap other warps' evaluation.
template <int MODE, bool DL32, bool FUSED, bool MANY, int EDGES>
__global__ void __launch_bounds__(kWarpsPerCta * 32, batch_min_blocks(MODE, DL32, MANY))
    k_eval_batch(DecideArgs a, int bin, int warp_bytes) {
    extern __shared__ __align__(16) unsigned char bsm[];
    using BW = BatchWarpT<EDGES>;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    BW &W = *reinterpret_cast<BW *>(bsm + (size_t)wid * warp_bytes);
    unsigned *dcnt = reinterpret_cast<unsigned *>(bsm + (size_t)wid * warp_bytes + sizeof(BW));
    const ModelDev &md = a.md;
    const int B = md.B;
    int *dlist = reinterpret_cast<int *>(dcnt + B);
    if (MODE == 1) {
        for (int i = lane; i < B; i += 32) dcnt[i] = 0u;
        __syncwarp();
    }
    Counts c;
    const int64_t gw = (int64_t)blockIdx.x * nwarps + wid, nw = (int64_t)gridDim.x * nwarps;
    if constexpr (!FUSED) {
        const Mover *mlist = a.movers + a.mbase[bin];
        const int64_t count = *(volatile unsigned *)&a.mcount[bin];
        const int64_t nbatch = (count + 31) >> 5;
        for (int64_t bt = gw; bt < nbatch; bt += nw) {
            const int64_t first_i = bt << 5;
            const int nv = (int)(count - first_i < 32 ? count - first_i : 32);
            Mover mv{0, -1, 0ull};
            if (lane < nv) mv = mlist[first_i + lane];
            batch_movers<MODE, DL32, EDGES>(a, W, dcnt, dlist, nv, mv.v, mv.s, mv.w2, c);
        }
        flush_counts_warp(md, c, 0ull);
    } else {
        const int32_t *vl = a.vlist[bin];
        const int64_t vcount = a.vcount[bin];
        const int64_t nvb = (vcount + 31) >> 5;
        unsigned long long medges = 0;
        int q0v = 0, q0s = -1, q1v = 0, q1s = -1, nq = 0;
        uint64_t q0w = 0, q1w = 0;
        for (int64_t vb = gw;; vb += nw) {
            const bool more = vb < nvb;
            if (more) {
                const int64_t i = (vb << 5) + lane;
                bool mover = false;
                int pv = 0, ps = 0;
                uint64_t pw = 0;
                if (i < vcount) {
                    pv = vl[i];
                    const Proposal p = propose_vertex(a.g, md, a.seed, a.sweep_id, pv);
                    if (p.s == p.r) {
                        c.proposed++;
                    } else {
                        mover = true;
                        ps = p.s;
                        pw = p.w2;
                        medges += (unsigned long long)p.k;
                    }
                }
                const unsigned mask = __ballot_sync(0xffffffffu, mover);
                const int cnt = __popc(mask);
                // queue positions nq .. nq + cnt - 1 take the new movers in lane order
                const int r0 = lane - nq, r1 = 32 + lane - nq;
                const bool t0 = r0 >= 0 && r0 < cnt, t1 = r1 >= 0 && r1 < cnt;
                const int src0 = t0 ? nth_set_bit(mask, r0) : lane, src1 = t1 ? nth_set_bit(mask, r1) : lane;
                const int v0 = __shfl_sync(0xffffffffu, pv, src0), s0 = __shfl_sync(0xffffffffu, ps, src0);
                const uint64_t w0 = __shfl_sync(0xffffffffu, pw, src0);
                const int v1 = __shfl_sync(0xffffffffu, pv, src1), s1 = __shfl_sync(0xffffffffu, ps, src1);
                const uint64_t w1 = __shfl_sync(0xffffffffu, pw, src1);
                if (t0) { q0v = v0; q0s = s0; q0w = w0; }
                if (t1) { q1v = v1; q1s = s1; q1w = w1; }
                nq += cnt;
            }
            while (nq >= 32 || (!more && nq > 0)) {
                const int nv = nq < 32 ? nq : 32;
                const int v = q0v, s = q0s;
                const uint64_t w2 = q0w;
                q0v = q1v; q0s = q1s; q0w = q1w;
                nq -= nv;
                batch_movers<MODE, DL32, EDGES>(a, W, dcnt, dlist, nv, v, s, w2, c);
            }
            if (!more) break;
        }
        flush_counts_warp(md, c, medges);
    }
}

// ---------------------------------------------------------------------------
// Sequential part of the hybrid pass (one CTA).  The h highest-degree
// vertices, in order, each decided against the current (b, M) with the exact
// evaluation (fixed-point Delta L, FP64 Hastings and test) and, when accepted,
// applied at once: the cells of its edges, the degrees of r and s, the
// labels.  The prefix rows P are rebuilt after this kernel; here the inverse
// CDF of the proposal scans row u (then column u) of M directly.
constexpr int kHybThreads = 256;

__device__ __forceinline__ int cta_first_above(const int32_t *M, int B, int u, bool column, uint32_t t, int *s_out,
                                               uint32_t *s_carry) {
    // smallest c with sum_{c' <= c} (row u or column u of M)[c'] > t
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    __shared__ uint32_t wsum[kHybThreads / 32];
    if (tid == 0) {
        *s_out = B - 1;
        *s_carry = 0;
    }
    __syncthreads();
    for (int c0 = 0; c0 < B; c0 += kHybThreads) {
        const int c = c0 + tid;
        const uint32_t x = c < B ? (uint32_t)(column ? M[(size_t)c * B + u] : M[(size_t)u * B + c]) : 0u;
        uint32_t incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        uint32_t before = *s_carry, total = 0;
        for (int q = 0; q < kHybThreads / 32; ++q) {
            before += q < w ? wsum[q] : 0u;
            total += wsum[q];
        }
        const uint32_t p = before + incl;
        const bool found = c < B && p > t && p - x <= t;
        __syncthreads();
        if (found) *s_out = c;
        if (tid == 0) *s_carry += total;
        const int any = __syncthreads_or(found ? 1 : 0);
        if (any) break;
    }
    __syncthreads();
    return *s_out;
}

__global__ void __launch_bounds__(kHybThreads) k_hybrid_seq(DecideArgs a, const int32_t *__restrict__ order, int h,
                                                            int32_t *M, int32_t *dout, int32_t *din, int32_t *dsum,
                                                            double *rcp, float *rcp32, int32_t *b, int32_t *bnew) {
    extern __shared__ unsigned hsm[];
    const ModelDev &md = a.md;
    const GraphDev &g = a.g;
    const int B = md.B, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    unsigned *cnt = hsm;
    int *list = reinterpret_cast<int *>(hsm + B);
    __shared__ int s_nl, s_self, s_u, s_mode, s_s, s_dec, s_pick;
    __shared__ uint32_t s_t, s_carry;
    __shared__ unsigned long long s_w2;
    __shared__ __int128 r_dl[kHybThreads / 32];
    __shared__ double r_fb[kHybThreads / 32], r_pf[kHybThreads / 32], r_pb[kHybThreads / 32];
    for (int i = tid; i < B; i += kHybThreads) cnt[i] = 0u;
    if (tid == 0) {
        s_nl = 0;
        s_self = 0;
    }
    Counts c;
    __syncthreads();
    for (int i = 0; i < h; ++i) {
        const int v = order[i];
        const int r = b[v];
        const int o0 = g.op[v], kout = g.op[v + 1] - o0, i0 = g.ip[v], kin = g.ip[v + 1] - i0, k = kout + kin;
        if (k == 0) {
            if (tid == 0) write_trace(a, v, r, 0, 0.0, 0.0);
            continue;
        }
        // the proposal, as in propose_vertex, against the current state
        if (tid == 0) {
            const U64x4 wd = philox4x64_10(a.sweep_id, (uint64_t)v, 0, 0, a.seed, 0);
            const int j = (int)draw_below(wd.x, (uint64_t)k);
            const int nb = j < kout ? g.oc[o0 + j] : g.ic[i0 + j - kout];
            const int u = b[nb];
            const int64_t y = draw_below(wd.y, (uint64_t)((int64_t)dsum[u] + B));
            s_w2 = wd.z;
            s_u = u;
            if (y < B) {
                s_mode = 0;
                s_s = (int)y;
            } else if (y - B < dout[u]) {
                s_mode = 1;
                s_t = (uint32_t)(y - B);
            } else {
                s_mode = 2;
                s_t = (uint32_t)(y - B - dout[u]);
            }
        }
        __syncthreads();
        int s = s_s;
        if (s_mode != 0) s = cta_first_above(M, B, s_u, s_mode == 2, s_t, &s_pick, &s_carry);
        if (s == r) {
            if (tid == 0) {
                write_trace(a, v, r, 1, 0.0, 0.0);
                c.proposed++;
            }
            __syncthreads();
            continue;
        }
        // v's neighbour blocks: direct-mapped counts ko | ki << 16
        for (int e = tid; e < k; e += kHybThreads) {
            const bool is_out = e < kout;
            const int nb = is_out ? g.oc[o0 + e] : g.ic[i0 + e - kout];
            if (nb == v) {
                if (is_out) atomicAdd(&s_self, 1);
                continue;
            }
            const int t = b[nb];
            if (atomicAdd(&cnt[t], is_out ? 1u : 0x10000u) == 0u) list[atomicAdd(&s_nl, 1)] = t;
        }
        __syncthreads();
        VertexCtx x;
        x.v = v;
        x.r = r;
        x.s = s;
        x.Kout = kout;
        x.Kin = kin;
        x.self = s_self;
        x.k = k;
        x.ko_r = (int)(cnt[r] & 0xffffu);
        x.ki_r = (int)(cnt[r] >> 16);
        x.ko_s = (int)(cnt[s] & 0xffffu);
        x.ki_s = (int)(cnt[s] >> 16);
        const int nl = s_nl;
        __int128 dl = 0;
        double fb = 0.0, pf = 0.0, pb = 0.0;
        for (int e = tid; e < nl; e += kHybThreads) {
            const int t = list[e];
            if (t == r || t == s) continue;
            const unsigned cc = cnt[t];
            entry_exact_all(md, x, t, (int)(cc & 0xffffu), (int)(cc >> 16), dl, fb, pf, pb);
        }
        if (tid < 8) special_terms(md, x, tid, dl, fb);
        dl = warp_sum_128(dl);
        fb = warp_sum(fb);
        pf = warp_sum(pf);
        pb = warp_sum(pb);
        if (lane == 0) {
            r_dl[w] = dl;
            r_fb[w] = fb;
            r_pf[w] = pf;
            r_pb[w] = pb;
        }
        __syncthreads();
        if (tid == 0) {
            __int128 dlt = 0;
            double fbt = 0.0, pft = 0.0, pbt = 0.0;
            for (int q = 0; q < kHybThreads / 32; ++q) {
                dlt += r_dl[q];
                fbt += r_fb[q];
                pft += r_pf[q];
                pbt += r_pb[q];
            }
            CornerVals cv;
            cv.Mrr = Mat(md, r, r);
            cv.Mss = Mat(md, s, s);
            cv.Mrs = Mat(md, r, s);
            cv.Msr = Mat(md, s, r);
            cv.dr = dsum[r];
            cv.ds = dsum[s];
            corner_hastings_exact(x, cv, B, pft, pbt);
            const Exact e = exact_decision(a.beta, dlt, fbt, pft, pbt, s_w2);
            count_exact(c, e.accept, e.margin, 0);
            write_trace(a, v, s, 1 | (e.accept ? 2 : 0) | (e.margin ? 4 : 0), e.dH, e.logA);
            s_dec = e.accept ? 1 : 0;
        }
        __syncthreads();
        if (s_dec) {
            // apply the move: the cells of v's edges, then degrees and labels
            for (int e = tid; e < kout; e += kHybThreads) {
                const int wv = g.oc[o0 + e];
                const int tw = wv == v ? r : b[wv], tn = wv == v ? s : b[wv];
                atomicAdd(&M[(size_t)r * B + tw], -1);
                atomicAdd(&M[(size_t)s * B + tn], 1);
            }
            for (int e = tid; e < kin; e += kHybThreads) {
                const int wv = g.ic[i0 + e];
                if (wv == v) continue;
                const int tw = b[wv];
                atomicAdd(&M[(size_t)tw * B + r], -1);
                atomicAdd(&M[(size_t)tw * B + s], 1);
            }
            __syncthreads();
            if (tid == 0) {
                dout[r] -= kout;
                dout[s] += kout;
                din[r] -= kin;
                din[s] += kin;
                const int qs[2] = {r, s};
                for (int q = 0; q < 2; ++q) {
                    const int bq = qs[q];
                    dsum[bq] = dout[bq] + din[bq];
                    rcp[bq] = 1.0 / ((double)dout[bq] + (double)din[bq] + (double)B);
                    rcp32[bq] = 1.0f / ((float)dout[bq] + (float)din[bq] + (float)B);
                }
                b[v] = s;
                bnew[v] = s;
            }
        }
        __syncthreads();
        for (int e = tid; e < nl; e += kHybThreads) cnt[list[e]] = 0u;
        if (tid == 0) {
            s_nl = 0;
            s_self = 0;
        }
        __syncthreads();
    }
    if (tid == 0) flush_counts(md, c);
}

__global__ void k_dxlogx32(const int32_t *__restrict__ x, const int32_t *__restrict__ k, int n, float *__restrict__ val,
                           float *__restrict__ am) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float a = 0.0f;
    val[i] = dxlogx32(x[i], k[i], a);
    am[i] = a;
}

__global__ void k_mark_skip(const int32_t *__restrict__ order, int h, int n, uint8_t *__restrict__ skip) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) skip[i] = 0;
}

__global__ void k_mark_skip2(const int32_t *__restrict__ order, int h, uint8_t *__restrict__ skip) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < h; i += gridDim.x * blockDim.x) skip[order[i]] = 1;
}

int sm_count() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

}  // namespace

// Graphs with at least this many edges run the three degree groups' kernels
// on three streams: none of them fills the chip (13 to 35% of the warps
// active at 200k vertices), and each ends in a tail.  One stream and three, a
// decision pass: 200k vertices, 4M edges at B = 223 223 and 200 us, at 4096
// 507 and 426, at 65,536 1231 and 903; 100k vertices, 1.6M edges 126 and 99.
// At 2^18 edges (10,000 vertices, exact form) the fork costs what it gains:
// 118 and 120 us.
static constexpr int64_t kSideStreamEdges = int64_t(1) << 19;
static constexpr int64_t kSideFirstGroup = 8192;

// three streams for kernels that may run together: the model's own one (for
// the longest) and its side streams, forked here and joined by join_side (all
// the model's own on smaller graphs)
int fork_side(sbp_model *m, cudaStream_t st[3]) {
    st[0] = st[1] = st[2] = m->stream;
    if (m->g->m < kSideStreamEdges) return SBP_OK;
    // (a call that failed half way left what it had made)
    for (int i = 0; i < 2; ++i) {
        if (!m->side[i]) SBP_CUDA(cudaStreamCreateWithFlags(&m->side[i], cudaStreamNonBlocking));
        if (!m->join_ev[i]) SBP_CUDA(cudaEventCreateWithFlags(&m->join_ev[i], cudaEventDisableTiming));
    }
    if (!m->fork_ev) SBP_CUDA(cudaEventCreateWithFlags(&m->fork_ev, cudaEventDisableTiming));
    SBP_CUDA(cudaEventRecord(m->fork_ev, m->stream));
    for (int i = 0; i < 2; ++i) SBP_CUDA(cudaStreamWaitEvent(m->side[i], m->fork_ev, 0));
    st[0] = m->side[1];
    st[1] = m->side[0];
    return SBP_OK;
}

int join_side(sbp_model *m) {
    if (m->g->m < kSideStreamEdges || !m->fork_ev) return SBP_OK;
    int rc = SBP_OK;  // both are joined, whatever the first gives
    for (int i = 0; i < 2; ++i) {
        cudaError_t e = cudaEventRecord(m->join_ev[i], m->side[i]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(m->stream, m->join_ev[i], 0);
        else cudaStreamSynchronize(m->side[i]);
        if (e != cudaSuccess) rc = cuda_fail(e, "joining the side streams");
    }
    return rc;
}

ModelDev model_dev(sbp_model *m) {
    ModelDev d;
    d.B = m->B;
    d.n = (int32_t)m->g->n;
    d.m = m->g->m;
    d.b = m->b;
    d.bnew = m->bnew;
    d.M = m->M;
    d.P = m->P;
    d.Pc = m->Pc;
    d.pstep = (2 * m->B + 31) / 32;
    d.dout = m->dout;
    d.din = m->din;
    d.rcp = m->rcp;
    d.rcp32 = m->rcp32;
    d.dsum = m->dsum;
    d.T = m->T;
    d.XT = m->XT;
    d.sparse = m->dense ? 0 : 1;
    d.rp = m->sp.rp;
    d.re = m->sp.slack ? m->sp.re : m->sp.rp + 1;
    d.cp = m->sp.cp;
    d.ce = m->sp.slack ? m->sp.ce : m->sp.cp + 1;
    d.hoff = m->sp.hoff;
    d.rc = m->sp.rc;
    d.cr = m->sp.cr;
    d.rv = m->sp.rv;
    d.cv = m->sp.cv;
    d.rpre = m->sp.rpre;
    d.cpre = m->sp.cpre;
    d.rpc = m->sp.rpc;
    d.cpc = m->sp.cpc;
    d.hkv = m->sp.hkv;
    d.status = m->status;
    d.counters = m->counters;
    d.items = nullptr;  // set by the nodal pass only
    d.cap_items = 0;
    d.nbo = nullptr;
    d.nbi = nullptr;
    return d;
}

namespace {

// The CTA kernel's neighbour table (cap slots of 16 bytes): in shared memory
// while it fits, else a slice per CTA of a global scratch the model keeps
// (at most 1 GB, fewer CTAs for very large tables).
size_t cta_table_bytes(int cap, int sms, int *grid) {
    const size_t bytes = (size_t)cap * 16;
    *grid = sms * 4;
    if (bytes <= 160 * 1024) return 0;
    const size_t per_grid = std::max<size_t>(1, (size_t(1) << 30) / bytes);
    if ((size_t)*grid > per_grid) *grid = (int)per_grid;
    return bytes * (size_t)*grid;
}

// log2 of the slots that hold a hub's distinct neighbour blocks at a load of
// at most 0.8
int hub_cap_log2(const sbp_graph *g, int64_t B) {
    const int64_t dmax = g->max_deg < B ? g->max_deg : B;
    const int64_t need = dmax + dmax / 4 + 2;
    int cap_log2 = 6;
    while ((int64_t(1) << cap_log2) < need) ++cap_log2;
    return cap_log2;
}

int cta_table(sbp_model *m, int cap, int sms, int *grid, size_t *smem, unsigned long long **gtab) {
    const size_t need = cta_table_bytes(cap, sms, grid);
    *gtab = nullptr;
    *smem = (size_t)cap * 16;
    if (need == 0) return SBP_OK;
    *smem = 0;
    if (m->cta_tab_bytes < need) {
        model_free(m->cta_tab, m->stream);
        m->cta_tab = nullptr;
        m->cta_tab_bytes = 0;
        if (model_alloc((void **)&m->cta_tab, need, m->stream) != cudaSuccess) {
            cudaGetLastError();
            return fail(SBP_ENOMEM, "nodal pass: no device memory for the neighbour tables");
        }
        m->cta_tab_bytes = need;
    }
    *gtab = m->cta_tab;
    return SBP_OK;
}

// Warps of a CTA of the kernels with direct-mapped counts: half as many where
// eight warps' counts would leave one CTA an SM (B > 1022).
int direct_warps(int B) { return (2 * B + 4) * 4 * kWarpsPerCta <= 64 * 1024 ? kWarpsPerCta : kWarpsPerCta / 2; }

// the evaluation kernels of the three degree groups: after k_propose, or
// (FUSED) drawing the proposals themselves
template <bool DL32, bool FUSED>
int launch_groups(sbp_model *m, const DecideArgs &a, int sms, const cudaStream_t st[3]) {
    const sbp_graph *g = m->g;
    const int B = m->B;
    // one launch of k_eval_table over list `bin`, tables of 2^cap_log2 slots
    auto tables = [&](int bin, int cap_log2, cudaStream_t on) -> int {
        const int cap = 1 << cap_log2;
        const size_t smem = (size_t)kWarpsPerCta * cap * 10;
        const size_t fixed = (size_t)kWarpsPerCta * (kTableQueue * 8 + 16) + 1024;  // static, and the system's
        const int per_sm = std::max(1, std::min(SBP_DECIDE_MIN_BLOCKS, (int)((size_t)228 * 1024 / (smem + fixed))));
        auto go = [&](auto kern) -> int {
            SBP_TRY(ensure_dyn_smem((const void *)kern, smem));
            kern<<<sms * per_sm, kWarpsPerCta * 32, smem, on>>>(a, bin, cap, cap_log2);
            SBP_LAUNCHED();
            return SBP_OK;
        };
        return m->dense ? go(k_eval_table<DL32, false>) : go(k_eval_table<DL32, true>);
    };
    // movers with k > 128: per-warp direct-mapped counts while B is small; at
    // larger B per-warp tables by degree class (each holds its class's
    // distinct blocks at a load of at most 0.8), one CTA per mover above
    // kWideDeg.  One table size for the whole group, set by the largest hub,
    // had sent all of it to the CTA kernel.
    if (g->bin[4] > g->bin[3] && !a.split_top) {
        const int warp_words = 2 * B + 4;
        const int nwarps = direct_warps(B);
        const size_t smem = (size_t)warp_words * 4 * nwarps;
        SBP_TRY(ensure_dyn_smem((const void *)k_eval_warp_direct<DL32, FUSED>, smem));
        k_eval_warp_direct<DL32, FUSED><<<sms * 4, nwarps * 32, smem, st[2]>>>(a, 2, warp_words);
        SBP_LAUNCHED();
    } else if (g->bin[4] > g->bin[3]) {
        if (g->n - g->bin[3] > g->n_mid + g->n_wide) {
            const int cap_log2 = hub_cap_log2(g, B);
            int grid;
            size_t smem;
            unsigned long long *gtab;
            SBP_TRY(cta_table(m, 1 << cap_log2, sms, &grid, &smem, &gtab));
            SBP_TRY(ensure_dyn_smem((const void *)k_eval_cta<DL32>, smem));
            k_eval_cta<DL32><<<grid, kBigThreads, smem, st[2]>>>(a, 4, 1 << cap_log2, cap_log2, gtab);
            SBP_LAUNCHED();
        }
        if (g->n_wide > 0) SBP_TRY(tables(3, 11, st[2]));
        if (g->n_mid > 0) SBP_TRY(tables(2, 10, st[0]));
    }
    // The batch kernels, with no more CTAs than the group has batches of 32
    // vertices.  Up to 10 KB a warp (B = 460), CTAs of eight warps, as many as
    // registers hold; three where shared memory holds two, the last ones
    // following and evening out the end (300,000 vertices with a heavy tail, B =
    // 330, FP32 form: 310 us, with two 355).  Above, as many CTAs of eight warps
    // as shared memory holds, if two (to B = 1500), else of four: 600,000
    // vertices of 40 edges, three CTAs of four warps and these, in us: B = 500
    // 643 and 425, 1000 561 and 422.
    auto batch = [&](auto kern, int bin, int min_blocks, size_t bytes, cudaStream_t on) -> int {
        const int wb = (int)((bytes + 15) / 16 * 16);
        auto held = [&](int nw) { return (int)(size_t(228) * 1024 / ((size_t)wb * nw + 1024)); };
        const int nw = wb <= 10 * 1024 || held(kWarpsPerCta) >= 2 ? kWarpsPerCta : kWarpsPerCta / 2;
        int ctas = min_blocks * kWarpsPerCta / nw;
        if (wb > 10 * 1024) ctas = std::min(ctas, held(nw));
        else if (held(nw) < 3) ctas = 3;
        const int64_t per_cta = 32 * nw, want = (g->bin[bin + 2] - g->bin[bin + 1] + per_cta - 1) / per_cta;
        const size_t smem = (size_t)wb * nw;
        SBP_TRY(ensure_dyn_smem((const void *)kern, smem));
        kern<<<(int)std::min<int64_t>(want, (int64_t)sms * ctas), nw * 32, smem, on>>>(a, bin, wb);
        SBP_LAUNCHED();
        return SBP_OK;
    };
    // The exact form's budgets (FP32 form's, own): a long pass over the first
    // group wants the warps; so does one over the second at few blocks, in us:
    // 300,000 vertices with a heavy tail, B = 50 (first group's budget) 194 and
    // 227, 307 and 349, 200,000 1238 and 1193 (three sweeps); 600,000, B = 50
    // (second group's) 529 and 656, of 80 edges 511 and 546, of 40 355 and 336.
    constexpr bool kTwo = !DL32;
    const bool many0 = g->n >= (int64_t(1) << 18), many1 = B <= 100 && g->m >= 10 * (int64_t(1) << 20);
    // movers with k <= 32: batches of 32 per warp
    if (g->bin[2] > g->bin[1]) {
        constexpr int E = kBatchEdges0;
        const size_t bytes = sizeof(BatchWarpT<E>);
        if (kTwo && many0)
            SBP_TRY(batch(k_eval_batch<0, DL32, FUSED, kTwo, E>, 0, batch_min_blocks(0, DL32, true), bytes, st[0]));
        else
            SBP_TRY(batch(k_eval_batch<0, DL32, FUSED, false, E>, 0, batch_min_blocks(0, DL32, false), bytes, st[0]));
    }
    // movers with 33 <= k <= 128: batches with direct-mapped counts while B is
    // small, otherwise one warp each with a 256-slot table
    if (g->bin[3] > g->bin[2]) {
        if (B <= kDirectMaxB) {
            constexpr int E = kBatchEdges, F = kBatchFewer;
            const size_t bytes = 4 * (size_t)B + 4 * kWarpDeg;
            const int few = batch_min_blocks(1, DL32, false);
            if (kTwo && many1)
                SBP_TRY(batch(k_eval_batch<1, DL32, FUSED, kTwo, E>, 1, batch_min_blocks(1, DL32, true),
                              bytes + sizeof(BatchWarpT<E>), st[1]));
            else if ((kTwo || !m->dense) && B >= 64 && B <= 320)
                SBP_TRY(batch(k_eval_batch<1, DL32, FUSED, false, F>, 1, few, bytes + sizeof(BatchWarpT<F>), st[1]));
            else
                SBP_TRY(batch(k_eval_batch<1, DL32, FUSED, false, E>, 1, few, bytes + sizeof(BatchWarpT<E>), st[1]));
        } else {
            SBP_TRY(tables(1, 8, st[1]));
        }
    }
    return SBP_OK;
}

// the movers the FP32 test left undecided (all of them when a trace is
// asked for): a CTA each, aggregated again and decided by the exact
// evaluation, after the three groups' kernels
template <bool DL32>
int launch_recheck(sbp_model *m, const DecideArgs &a0, int sms) {
    const sbp_graph *g = m->g;
    DecideArgs a = a0;
    a.force_exact = 1;
    const int cap_log2 = hub_cap_log2(g, m->B), cap = 1 << cap_log2;
    int grid;
    size_t smem;
    unsigned long long *gtab;
    SBP_TRY(cta_table(m, cap, sms, &grid, &smem, &gtab));
    SBP_TRY(ensure_dyn_smem((const void *)k_eval_cta<DL32>, smem));
    k_eval_cta<DL32><<<grid, kBigThreads, smem, m->stream>>>(a, kRecheck, cap, cap_log2, gtab);
    SBP_LAUNCHED();
    return SBP_OK;
}

// Whether a pass over the vertices of `a` takes k_eval_small, which gives
// every mover a warp: up to the most vertices at which it was nowhere slower
// than the groups' kernels, by what these have to do.
//   - Only the group of up to 32 edges: one kernel with 32 movers a warp.
//   - More groups: a kernel each, one after another below 2^19 edges.  The
//     second group's takes 30 to 70 us as soon as a few warps have a batch of
//     its movers; three hubs, or hundreds of rows above 128 edges, do not.
//   - From 2^19 edges they run on three streams, where the top group's rows
//     are the long ones; rows of hundreds of edges have a warp each there too,
//     with twice the warps, and win from some 2^21 edges on (the line: 3 x 2^19).
//   - B > 1022: half the warps here, none lost there in the first group; with a
//     second and a third group those cost more (B = 1500 and 2048, 100 vertices
//     of 50 edges and 100 of 300 among 120,000 edges, 30,000 vertices 145, 111,
//     40,000 162, 147; a heavy tail and 390,000 edges, 25,000 168, 93, 40,000
//     172, 138; the full run of 20,900 such vertices 58.1 ms, 48.7).
//   - From 2^19 to 3 x 2^18 edges and beyond 40,000 vertices a heavy tail would
//     gain (48,395 vertices, 598,074 edges at B = 72, labels set and a sweep 295,
//     273), a hundred long rows lose more (54,000, 528,000 at B = 72, 59, 95).
// Both sides in us (groups, small; labels near the planted ones, B = 4 / 1000;
// B = 2048): only the first group, 6000 vertices 27, 28 / 35, 34; 34, 36; at
// 20,000 42, 40 / 53, 60; 57, 83; at 60,000 50, 77 / 65, 109; 75, 193.  More
// groups, 6 edges a vertex and three hubs of 300, 20,000 vertices 51, 42 /
// 66, 56; 58, 83; at 30,000 54, 52 / 70, 69; 74, 112; at 60,000 62, 76 / 81,
// 107; 87, 187; 100 vertices of 40 among them, 40,000 82, 63 / 133, 83; 137,
// 139; 20 edges a vertex, 20,000 56, 42 / 97, 57; 95, 80, 40,000 71, 62 / 96, 77;
// 102, 130, 60,000 61, 77 / 96, 103; 98, 168; 32 edges a vertex, 20,000 71, 41 /
// 111, 52; 114, 75, 40,000 (2^19.3 edges) 48, 61 / 68, 75; 81, 120, with a heavy
// tail 70, 59 / 129, 80; 128, 124.
bool small_pass(const sbp_graph *g, const DecideArgs &a, int B) {
    const int64_t n = a.vcount[0] + a.vcount[1] + a.vcount[2];
    const bool half = direct_warps(B) < kWarpsPerCta;
    if (a.vcount[1] + a.vcount[2] == 0) return n <= (half ? 2500 : 5000);
    if (g->m < kSideStreamEdges && a.vcount[1] >= 64) return n <= (half && a.vcount[2] < 64 ? 20000 : 40000);
    if (g->m < kSideStreamEdges) return n <= (half ? 10000 : 22000);
    if (!half && a.vcount[2] >= 64 && g->m <= 3 * (int64_t(1) << 18)) return n <= 40000;
    return g->m <= 3 * (int64_t(1) << 19) && n <= (half ? 6000 : 20000);
}

template <bool DL32>
int launch_small(sbp_model *m, const DecideArgs &a, int sms) {
    const int warp_words = 2 * m->B + 4;
    const int nwarps = direct_warps(m->B);
    const size_t smem = (size_t)warp_words * 4 * nwarps;
    SBP_TRY(ensure_dyn_smem((const void *)k_eval_small<DL32>, smem));
    const int64_t n = a.vcount[0] + a.vcount[1] + a.vcount[2];
    const int64_t ctas = (n + nwarps - 1) / nwarps;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ctas, sms * 2));
    k_eval_small<DL32><<<grid, nwarps * 32, smem, m->stream>>>(a, warp_words);
    SBP_LAUNCHED();
    return SBP_OK;
}

template <bool DL32>
int launch_evals(sbp_model *m, const DecideArgs &a, int sms, bool fused) {
    cudaStream_t st[3] = {m->stream, m->stream, m->stream};
    // One group alone has nothing to run beside it (a sweep of 200k vertices of
    // 10 edges lost 10 us to the fork), and the first group's kernel on few
    // vertices is over in 7 us (two sweeps of 60,000 vertices of 67 edges, a
    // handful of them in it, at B = 1000: 611 us forked, 548 not).
    // (the top group's classes at large B are kernels of their own.)
    const sbp_graph *g = m->g;
    const int64_t *vc = a.vcount;
    const bool several = (vc[1] > 0 && vc[2] > 0) || (vc[0] >= kSideFirstGroup && vc[1] + vc[2] > 0) ||
                         (a.split_top && (g->n_mid > 0) + (g->n_wide > 0) + (vc[2] > g->n_mid + g->n_wide) > 1);
    if (several) SBP_TRY(fork_side(m, st));
    const int rc = fused ? launch_groups<DL32, true>(m, a, sms, st) : launch_groups<DL32, false>(m, a, sms, st);
    const int rj = several ? join_side(m) : SBP_OK;  // joined on every path
    if (rc != SBP_OK) return rc;
    if (rj != SBP_OK) return rj;
    return launch_recheck<DL32>(m, a, sms);
}

// at most one item per vertex plus one per kMoveChunk edge ends
int64_t most_items(const sbp_graph *g) { return g->n + (2 * g->m) / kMoveChunk + 1; }

}  // namespace

// the mover lists, the accepted-move list, the hybrid pass's flags, the hubs'
// tables
size_t pass_bytes(const sbp_graph *g, int64_t B) {
    int grid;
    return 2 * (size_t)g->n * sizeof(Mover) + (size_t)most_items(g) * sizeof(int2) + (size_t)g->n +
           cta_table_bytes(1 << hub_cap_log2(g, std::min<int64_t>(B, 1 << 24)), sm_count(), &grid);  // (B is below that)
}

int launch_decide(sbp_model *m, uint64_t sweep_id, int64_t v_begin, int64_t v_end, const sbp_vertex_trace *trace) {
    const sbp_graph *g = m->g;
    if (!m->movers) {
        // the degree groups' lists (n entries) and the recheck list (n more)
        if (model_alloc(&m->movers, (size_t)(g->n > 0 ? 2 * g->n : 1) * sizeof(Mover), m->stream) != cudaSuccess ||
            model_alloc((void **)&m->mcount, kMoverLists * sizeof(unsigned), m->stream) != cudaSuccess) {
            cudaGetLastError();
            return fail(SBP_ENOMEM, "cudaMalloc failed for the mover lists");
        }
    }
    if (!m->items) {
        const int64_t cap = most_items(g);
        if (model_alloc((void **)&m->items, (size_t)cap * sizeof(int2), m->stream) != cudaSuccess) {
            cudaGetLastError();
            return fail(SBP_ENOMEM, "cudaMalloc failed for the accepted-move list");
        }
        m->cap_items = cap;
    }
    // the list holds every accepted move only while the ranges decided since
    // the last commit are disjoint
    for (const auto &rg : m->decided)
        if (v_begin < rg.second && rg.first < v_end) m->list_ok = false;
    m->decided.emplace_back(v_begin, v_end);
    DecideArgs a;
    a.g = g->dev();
    a.md = model_dev(m);
    a.md.items = m->items;
    a.md.cap_items = m->cap_items;
    const int64_t h_seq = std::min<int64_t>(m->p.hybrid_h, g->n);
    if (h_seq > 0 && m->dense && v_begin == 0 && v_end == g->n) {
        m->nb_ok = false;  // the sequential part moves vertices in place
    } else {
        if (!m->nb_ok) SBP_TRY(nb_rows_rebuild(m));
        if (m->nb_ok) {
            a.md.nbo = m->nbo;
            a.md.nbi = m->nbi;
        }
    }
    a.v_begin = v_begin;
    a.v_end = v_end;
    a.movers = static_cast<Mover *>(m->movers);
    a.mcount = m->mcount;
    // list capacities: the sizes of the degree groups
    a.mbase[0] = 0;
    a.mbase[1] = g->bin[2] - g->bin[1];
    a.mbase[2] = a.mbase[1] + (g->bin[3] - g->bin[2]);
    a.mbase[3] = a.mbase[2] + g->n_mid;
    a.mbase[4] = a.mbase[3] + g->n_wide;
    a.mbase[kRecheck] = g->n;
    a.force_exact = 0;
    a.seed = m->p.seed;
    a.sweep_id = sweep_id;
    a.beta = m->p.beta;
    a.beta32 = (float)m->p.beta;
    a.tr = trace ? *trace : sbp_vertex_trace{nullptr, nullptr, nullptr, nullptr};
    a.skip = nullptr;
    a.trace_on = (a.tr.s || a.tr.flags || a.tr.dH || a.tr.logA) ? 1 : 0;
    const int sms = sm_count();
    const int B = m->B;
    a.split_top = B > kDirectMaxB || g->max_deg >= 65536;
    if (B >= (1 << 24)) return fail(SBP_ESTATE, "nodal pass: B must be below 2^24");
    // hybrid pass: the sequential part first (full-range passes of a dense model)
    const int64_t h = std::min<int64_t>(m->p.hybrid_h, g->n);
    if (h > 0 && m->dense && v_begin == 0 && v_end == g->n) {
        if (g->max_deg >= 65536) return fail(SBP_ESTATE, "hybrid pass: degrees of 65536 or more are not supported");
        if (!m->skip) {
            if (model_alloc((void **)&m->skip, (size_t)g->n, m->stream) != cudaSuccess) {
                cudaGetLastError();
                return fail(SBP_ENOMEM, "device allocation failed for the hybrid pass");
            }
            m->skip_h = -1;
        }
        if (m->skip_h != (int32_t)h) {
            k_mark_skip<<<(int)std::min<int64_t>((g->n + 255) / 256, 1024), 256, 0, m->stream>>>(g->by_degree, (int)h,
                                                                                                 (int)g->n, m->skip);
            SBP_LAUNCHED();
            k_mark_skip2<<<(int)std::min<int64_t>((h + 255) / 256, 1024), 256, 0, m->stream>>>(g->by_degree, (int)h,
                                                                                               m->skip);
            SBP_LAUNCHED();
            m->skip_h = (int32_t)h;
        }
        const size_t smem = (size_t)B * 8;
        SBP_TRY(ensure_dyn_smem((const void *)k_hybrid_seq, smem));
        k_hybrid_seq<<<1, kHybThreads, smem, m->stream>>>(a, g->by_degree, (int)h, m->M, m->dout, m->din, m->dsum,
                                                          m->rcp, m->rcp32, m->b, m->bnew);
        SBP_LAUNCHED();
        SBP_TRY(launch_prefix(m));
        a.skip = m->skip;
    }

    // A full-range pass with no trace and no sequential part, whose degree
    // groups all take the direct-mapped kernels, draws the proposals inside
    // the evaluation kernels; any other pass proposes every vertex of its
    // range first (k_propose) and hands the movers over in lists.
    for (int i = 0; i < 3; ++i) {
        a.vlist[i] = g->order + g->bin[i + 1];
        a.vcount[i] = g->bin[i + 2] - g->bin[i + 1];
    }
    const bool fused = SBP_FUSED_PROPOSALS && v_begin == 0 && v_end == g->n && !a.skip && !a.trace_on &&
                       B <= kDirectMaxB && g->max_deg < 65536;
    if (fused && small_pass(g, a, B))
        return m->p.dl_fp32 ? launch_small<true>(m, a, sms) : launch_small<false>(m, a, sms);
    SBP_CUDA(cudaMemsetAsync(m->mcount, 0, kMoverLists * sizeof(unsigned), m->stream));
    if (!fused) {
        int64_t blocks = (v_end - v_begin + 255) / 256;
        if (blocks > (int64_t)sms * 8) blocks = (int64_t)sms * 8;
        if (blocks < 1) blocks = 1;
        k_propose<<<(int)blocks, 256, 0, m->stream>>>(a);
        SBP_LAUNCHED();
    }
    return m->p.dl_fp32 ? launch_evals<true>(m, a, sms, fused) : launch_evals<false>(m, a, sms, fused);
}

}  // namespace sbp

// Known-answer hook for the FP32 term of the precision form: val[i] =
// f(x[i] + k[i]) - f(x[i]) in FP32 and am[i] the magnitude its error bound
// is proportional to (host arrays).
extern "C" int sbp_dxlogx32_check(const int32_t *x, const int32_t *k, int32_t count, float *val, float *am) {
    using namespace sbp;
    if (count < 0 || count > (1 << 24) || (count > 0 && (!x || !k || !val || !am)))
        return fail(SBP_EINVAL, "sbp_dxlogx32_check: bad count or NULL array");
    for (int32_t i = 0; i < count; ++i)
        if (x[i] < 0 || (int64_t)x[i] + k[i] < 0 || (int64_t)x[i] + k[i] > INT32_MAX)
            return fail(SBP_EINVAL, "sbp_dxlogx32_check: need x >= 0 and 0 <= x + k < 2^31");
    if (count == 0) return SBP_OK;
    void *d = nullptr;
    SBP_CUDA(cudaMalloc(&d, (size_t)count * 16));
    int32_t *dx = static_cast<int32_t *>(d), *dk = dx + count;
    float *dv = reinterpret_cast<float *>(dk + count), *da = dv + count;
    cudaError_t e = cudaMemcpy(dx, x, (size_t)count * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dk, k, (size_t)count * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_dxlogx32<<<(count + 255) / 256, 256>>>(dx, dk, count, dv, da);
        count_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(val, dv, (size_t)count * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(am, da, (size_t)count * 4, cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess) return cuda_fail(e, "sbp_dxlogx32_check");
    return SBP_OK;
}
