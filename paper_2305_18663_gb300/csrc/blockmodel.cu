// blockmodel.cu -- the blockmodel from the assignment, and its update after
// a pass.
//
// Section II-A: M[r][s] counts the edges from block r to block s; the block
// degrees are its row and column sums.  Alg. 5: after every pass the moves
// are applied and the blockmodel is made consistent again: each edge with a
// moved end leaves its old (block, block) cell and enters the new one when
// the moved rows hold at most a quarter of the edges (a plan taken on the
// device), else M is recounted from the new assignment.  Both give the same
// integers.  The same kernels keep the block-labelled rows in step.
//
// Dense form (B <= dense_max_B): M is B x B int32, counted by an atomic
// histogram over the out-edges with the diagonal privatised per CTA.  P
// holds, per block u, the inclusive prefix of row u followed by dout_u plus
// the inclusive prefix of column u; the nodal and merge proposals search it.
// DL (Eq. 2) is reduced in a fixed order so it is reproducible bit for bit.
#include <algorithm>
#include <cmath>

#include "apply.cuh"

namespace sbp {
namespace {

constexpr int kThreads = 256;

// Atomic histogram of (b[src], b[dst]) over the out-edges, four
// consecutive edges per thread (16-byte loads, eight independent gathers in
// flight).  Diagonal counts (intra-block edges, the large majority) go to a
// per-CTA shared-memory copy of the diagonal first.
__device__ __forceinline__ void hist_add(int32_t *__restrict__ M, int *diag, int B, bool valid, int r, int t) {
    if (!valid) return;
    if (r == t) atomicAdd(&diag[r], 1);
    else atomicAdd(&M[(size_t)r * B + t], 1);
}

__global__ void __launch_bounds__(kThreads) k_hist_dense(GraphDev g, const int32_t *__restrict__ b,
                                                         int32_t *__restrict__ M, int B, const int32_t *__restrict__ skip) {
    if (skip && *skip == 1) return;
    extern __shared__ int diag[];
    for (int i = threadIdx.x; i < B; i += blockDim.x) diag[i] = 0;
    __syncthreads();
    const int64_t m4 = g.m >> 2;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int4 *es4 = reinterpret_cast<const int4 *>(g.esrc);
    const int4 *oc4 = reinterpret_cast<const int4 *>(g.oc);
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < m4; base += stride) {
        const int64_t q = base + threadIdx.x;
        const bool valid = q < m4;
        int4 s4 = make_int4(0, 0, 0, 0), d4 = make_int4(0, 0, 0, 0);
        if (valid) {
            s4 = es4[q];
            d4 = oc4[q];
        }
        int r0 = 0, r1 = 0, r2 = 0, r3 = 0, t0 = 0, t1 = 0, t2 = 0, t3 = 0;
        if (valid) {
            r0 = b[s4.x]; r1 = b[s4.y]; r2 = b[s4.z]; r3 = b[s4.w];
            t0 = b[d4.x]; t1 = b[d4.y]; t2 = b[d4.z]; t3 = b[d4.w];
        }
        hist_add(M, diag, B, valid, r0, t0);
        hist_add(M, diag, B, valid, r1, t1);
        hist_add(M, diag, B, valid, r2, t2);
        hist_add(M, diag, B, valid, r3, t3);
    }
    // the last m % 4 edges
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        const int64_t e = (m4 << 2) + threadIdx.x;
        const bool valid = e < g.m;
        const int r = valid ? b[g.esrc[e]] : 0, t = valid ? b[g.oc[e]] : 0;
        hist_add(M, diag, B, valid, r, t);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < B; i += blockDim.x)
        if (diag[i]) atomicAdd(&M[(size_t)i * B + i], diag[i]);
}

// one warp per block u
__global__ void __launch_bounds__(kThreads) k_prefix_dense(const int32_t *__restrict__ M, int B,
                                                           uint32_t *__restrict__ P, int32_t *__restrict__ dout,
                                                           int32_t *__restrict__ din, double *__restrict__ rcp,
                                                           float *__restrict__ rcp32, int32_t *__restrict__ dsum,
                                                           uint32_t *__restrict__ Pc, int pstep) {
    const int u = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (u >= B) return;
    prefix_block<true>(M, B, u, P, dout, din, rcp, rcp32, dsum, Pc, pstep);
}

// The same at many blocks (B >= kWidePrefixB), in four steps that read and
// write whole lines: one warp per block reads its column of M with a stride
// of B words (113 us at B = 4096, with a sector of 32 bytes for every count).
//   1. k_prefix_rows: a block per row, its prefix, dout, and its share of L;
//   2. k_col_sums: 32 columns times kColChunk rows per block, column sums;
//   3. k_prefix_cols: the same tiles, transposed through shared memory, the
//      column prefixes from the sums of the chunks above;
//   4. k_wide_finish: pivots, din, reciprocals, the column degrees' share of L.
// Prefix rows and DL at B = 4096: 179 -> 94 us (rows 41, sums 15, columns 28,
// finish 9; 64 MB read twice, 134 MB written).  The line: labels of a 200k-vertex
// graph set from outside and committed, few of them changed, take, with a warp
// per block and with these, 83 and 98 us at B = 1000, 98 and 104 at 1500, 110
// and 105 at 1600, 104 and 104 at 1800, 111 and 109 at 2000, 125 and 123 at
// 2500, 150 and 137 at 3000.
constexpr int kWidePrefixB = 1600;
constexpr int kColChunk = 256;
constexpr int kRowIn = 8;  // counts of a row in flight per thread

__global__ void __launch_bounds__(kThreads) k_prefix_rows(const int32_t *__restrict__ M, int B,
                                                          uint32_t *__restrict__ P, int32_t *__restrict__ dout,
                                                          const __int128 *__restrict__ T, int64_t XT,
                                                          DlPartial *__restrict__ partials) {
    __shared__ uint32_t wsum[kRowIn][kThreads / 32];
    __shared__ __int128 sfix[kThreads / 32];
    __shared__ double sfb[kThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __int128 fix = 0;
    double fb = 0.0;
    for (int u = blockIdx.x; u < B; u += gridDim.x) {
        uint32_t carry = 0;
        for (int c0 = 0; c0 < B; c0 += kRowIn * kThreads) {
            uint32_t x[kRowIn];
#pragma unroll
            for (int q = 0; q < kRowIn; ++q) {
                const int c = c0 + q * kThreads + threadIdx.x;
                x[q] = c < B ? (uint32_t)M[(size_t)u * B + c] : 0u;
            }
#pragma unroll
            for (int q = 0; q < kRowIn; ++q) {
                add_xlogx(T, XT, x[q], 1, fix, fb);
                x[q] = warp_incl_scan_u32(x[q]);
                if (lane == 31) wsum[q][wid] = x[q];
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kRowIn; ++q) {
                const uint32_t w = lane < kThreads / 32 ? wsum[q][lane] : 0u;
                const uint32_t before = __reduce_add_sync(0xffffffffu, lane < wid ? w : 0u);
                const int c = c0 + q * kThreads + threadIdx.x;
                if (c < B) P[(size_t)u * 2 * B + c] = carry + before + x[q];
                carry += __reduce_add_sync(0xffffffffu, w);
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            dout[u] = (int32_t)carry;
            add_xlogx(T, XT, carry, -1, fix, fb);
        }
    }
    fix = warp_sum_128(fix);
    fb = warp_sum(fb);
    if (lane == 0) {
        sfix[wid] = fix;
        sfb[wid] = fb;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < kThreads / 32; ++q) {
            fix += sfix[q];
            fb += sfb[q];
        }
        partials[blockIdx.x].fix = fix;
        partials[blockIdx.x].fb = fb;
    }
}

__global__ void __launch_bounds__(kThreads) k_col_sums(const int32_t *__restrict__ M, int B,
                                                       uint32_t *__restrict__ sums) {
    __shared__ uint32_t part[kThreads / 32][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int u = blockIdx.x * 32 + lane, c0 = blockIdx.y * kColChunk;
    uint32_t s = 0;
#pragma unroll 8
    for (int q = wid; q < kColChunk; q += kThreads / 32)
        if (u < B && c0 + q < B) s += (uint32_t)M[(size_t)(c0 + q) * B + u];
    part[wid][lane] = s;
    __syncthreads();
    if (wid == 0 && u < B) {
        for (int w = 1; w < kThreads / 32; ++w) s += part[w][lane];
        sums[(size_t)blockIdx.y * B + u] = s;
    }
}

__global__ void __launch_bounds__(kThreads) k_prefix_cols(const int32_t *__restrict__ M, int B,
                                                          const uint32_t *__restrict__ sums,
                                                          const int32_t *__restrict__ dout, uint32_t *__restrict__ P) {
    __shared__ uint32_t tile[kColChunk][33], first[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int u0 = blockIdx.x * 32, c0 = blockIdx.y * kColChunk;
    constexpr int kWarps = kThreads / 32;
#pragma unroll
    for (int q = 0; q < kColChunk / kWarps; ++q) {
        const int c = q * kWarps + wid;
        tile[c][lane] = c0 + c < B && u0 + lane < B ? (uint32_t)M[(size_t)(c0 + c) * B + u0 + lane] : 0u;
    }
    if (wid == 0) {
        const int u = u0 + lane;
        uint32_t s = u < B ? (uint32_t)dout[u] : 0u;
#pragma unroll 8
        for (int y = 0; y < (int)blockIdx.y; ++y) s += u < B ? sums[(size_t)y * B + u] : 0u;
        first[lane] = s;
    }
    __syncthreads();
    for (int q = wid; q < 32 && u0 + q < B; q += kWarps) {
        uint32_t p[kColChunk / 32];
#pragma unroll
        for (int t = 0; t < kColChunk / 32; ++t) p[t] = warp_incl_scan_u32(tile[t * 32 + lane][q]);
        uint32_t carry = first[q];
        uint32_t *out = P + (size_t)(u0 + q) * 2 * B + B + c0;
#pragma unroll
        for (int t = 0; t < kColChunk / 32; ++t) {
            if (c0 + t * 32 + lane < B) out[t * 32 + lane] = carry + p[t];
            carry += __shfl_sync(0xffffffffu, p[t], 31);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_wide_finish(const uint32_t *__restrict__ P, int B,
                                                          const int32_t *__restrict__ dout, int32_t *__restrict__ din,
                                                          double *__restrict__ rcp, float *__restrict__ rcp32,
                                                          int32_t *__restrict__ dsum, uint32_t *__restrict__ Pc,
                                                          int pstep, const __int128 *__restrict__ T, int64_t XT,
                                                          DlPartial *__restrict__ partials) {
    __shared__ __int128 sfix[kThreads / 32];
    __shared__ double sfb[kThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __int128 fix = 0;
    double fb = 0.0;
    const int u = blockIdx.x * (kThreads / 32) + wid;
    if (u < B) {
        const uint32_t *row = P + (size_t)u * 2 * B;
        const int pi = (lane + 1) * pstep - 1 < 2 * B - 1 ? (lane + 1) * pstep - 1 : 2 * B - 1;
        Pc[(size_t)u * 32 + lane] = row[pi];
        if (lane == 0) {
            const uint32_t o = (uint32_t)dout[u], i = row[2 * B - 1] - o;
            din[u] = (int32_t)i;
            rcp[u] = 1.0 / ((double)o + (double)i + (double)B);
            rcp32[u] = 1.0f / ((float)o + (float)i + (float)B);
            dsum[u] = (int32_t)(o + i);
            add_xlogx(T, XT, i, -1, fix, fb);
        }
    }
    if (lane == 0) {
        sfix[wid] = fix;
        sfb[wid] = fb;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < kThreads / 32; ++q) {
            fix += sfix[q];
            fb += sfb[q];
        }
        partials[blockIdx.x].fix = fix;
        partials[blockIdx.x].fb = fb;
    }
}

// Eq. 1 split form: sum over M of x ln x minus the degree terms, one
// partial per block, exact in fixed point inside the table
__global__ void __launch_bounds__(kThreads) k_dl_partial(const int32_t *__restrict__ M, int64_t BB,
                                                         const int32_t *__restrict__ dout,
                                                         const int32_t *__restrict__ din, int B,
                                                         const __int128 *__restrict__ T, int64_t XT,
                                                         DlPartial *__restrict__ partials) {
    __shared__ __int128 sfix[kThreads / 32];
    __shared__ double sfb[kThreads / 32];
    __int128 fix = 0;
    double fb = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < BB; i += stride) add_xlogx(T, XT, M[i], 1, fix, fb);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < B; i += stride) {
        add_xlogx(T, XT, dout[i], -1, fix, fb);
        add_xlogx(T, XT, din[i], -1, fix, fb);
    }
    fix = warp_sum_128(fix);
    fb = warp_sum(fb);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        sfix[wid] = fix;
        sfb[wid] = fb;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __int128 f = 0;
        double d = 0.0;
        for (int q = 0; q < kThreads / 32; ++q) {
            f += sfix[q];
            d += sfb[q];
        }
        partials[blockIdx.x].fix = f;
        partials[blockIdx.x].fb = d;
    }
}

// Eq. 2: DL = E h(B^2/E) + N ln B - L, h(x) = (1+x) ln(1+x) - x ln x.  The
// partials are summed in a fixed order (strided per thread, then a fixed
// tree), so the result is reproducible bit for bit.
constexpr int kFinalThreads = 1024;
__global__ void __launch_bounds__(kFinalThreads) k_dl_final(const DlPartial *__restrict__ partials, int np, int64_t E,
                                                            int64_t N, int B, double *__restrict__ dl) {
    __shared__ __int128 sfix[kFinalThreads / 32];
    __shared__ double sfb[kFinalThreads / 32];
    __shared__ double model;
    // the part without the counts (a chain of FP64 logarithms) on a thread of its own
    if (threadIdx.x == kFinalThreads - 1) model = dl_eq2(E, N, B, 0.0);
    __int128 f = 0;
    double d = 0.0;
    for (int i = threadIdx.x; i < np; i += kFinalThreads) {
        f += partials[i].fix;
        d += partials[i].fb;
    }
    f = warp_sum_128(f);
    d = warp_sum(d);
    if ((threadIdx.x & 31) == 0) {
        sfix[threadIdx.x >> 5] = f;
        sfb[threadIdx.x >> 5] = d;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        f = warp_sum_128(sfix[threadIdx.x]);
        d = warp_sum(sfb[threadIdx.x]);
        if (threadIdx.x == 0) dl[0] = model - (fix_to_double(f) + d);
    }
}

// commit plan (1 = update the counts from the moved vertices' rows, when
// they hold at most a quarter of the edges; 0 = recount) and, for a recount,
// the zeroed cells: every CTA derives the plan from the counters, CTA 0
// stores it for the kernels that follow
__global__ void k_commit_plan(const DevCounters *__restrict__ c, int64_t E, int32_t *__restrict__ flag,
                              int32_t *__restrict__ M, int64_t n) {
    const int plan = (c->acc_edges * 4ull <= (unsigned long long)E) ? 1 : 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) flag[0] = plan;
    if (plan != 0) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) M[i] = 0;
}

// Apply step of Alg. 5 on a dense M: every edge with a moved end leaves its
// old (block, block) cell and enters the new one.  An edge is visited once:
// through the out-row of its moved source, or through the in-row of its
// moved target when the source stayed.  Lanes take the edges of one row,
// four loads in flight per lane.
// Warps [0, n_big) take one vertex each of the largest-degree group (in
// descending degree, so the longest rows start first); the remaining warps
// take 32 consecutive vertex ids each and skip the ones of that group.
__global__ void __launch_bounds__(kThreads) k_delta_dense(GraphDev g, const int32_t *__restrict__ order, int big_begin,
                                                          int n_big, const int32_t *__restrict__ bnew,
                                                          const int32_t *__restrict__ bold, int32_t *__restrict__ M,
                                                          int B, const int32_t *__restrict__ flag) {
    if (*flag != 1) return;
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w < n_big) {
        const int v = order[big_begin + w];
        const int r = bold[v], s = bnew[v];
        if (r == s) return;
        delta_out_row(g.oc, g.op[v], g.op[v + 1], r, s, bnew, bold, M, B);
        delta_in_row(g.ic, g.ip[v], g.ip[v + 1], r, s, bnew, bold, M, B);
        return;
    }
    const int64_t base = (w - n_big) * 32;
    if (base >= g.n) return;
    const int64_t vv = base + lane;
    const bool moved = vv < g.n && bnew[vv] != bold[vv];
    unsigned mm = __ballot_sync(0xffffffffu, moved);
    while (mm) {
        const int q = __ffs(mm) - 1;
        mm &= mm - 1;
        const int v = (int)(base + q);
        const int o0 = g.op[v], o1 = g.op[v + 1], i0 = g.ip[v], i1 = g.ip[v + 1];
        if ((o1 - o0) + (i1 - i0) > kWarpDeg) continue;  // a warp of its own took it
        const int r = bold[v], s = bnew[v];
        delta_out_row(g.oc, o0, o1, r, s, bnew, bold, M, B);
        delta_in_row(g.ic, i0, i1, r, s, bnew, bold, M, B);
    }
}

// Adds d to cells[key] for every lane with key >= 0.  The lanes whose key
// equals that of the first lane holding one add together with one atomic
// (most edges of a moved vertex land on the same (block, block) cell); the
// other lanes add their own.  All lanes of the warp call it.
__device__ __forceinline__ void warp_cell_add(int32_t *cells, int key, int d) {
    const unsigned act = __ballot_sync(0xffffffffu, key >= 0);
    if (!act) return;
    const int lead = __ffs(act) - 1;
    const int k0 = __shfl_sync(0xffffffffu, key, lead);
    const unsigned same = __ballot_sync(0xffffffffu, key == k0);
    if ((int)(threadIdx.x & 31) == lead)
        atomicAdd(&cells[k0], d * __popc(same));
    else if (key >= 0 && key != k0)
        atomicAdd(&cells[key], d);
}

// One item of the accepted-move list, on a warp: a kMoveChunk-edge slice of
// the concatenated (out, in) row of a moved vertex, kItemIn chunks of 32
// edges in flight.  counts: the cells are updated; nbo (not NULL): the
// block-labelled rows too (the twin of each edge takes v's new label).
// Bound by the latency of its four dependent rounds of scattered loads: most
// items are the 40-odd edges of one vertex, so what counts is how many warps
// are in flight, not how many loads each has: 8 loads a lane at 48 registers
// and 4 blocks an SM against 2 at 32 and 8, three sweeps of a 1M-vertex graph
// took 3770 and 3670 us (4 loads, 6 blocks: 3677).
constexpr int kItemIn = 2;

__device__ __forceinline__ void delta_item(const GraphDev &g, int2 it, const int32_t *__restrict__ bnew,
                                           const int32_t *__restrict__ bold, int32_t *__restrict__ M, int B,
                                           bool counts, int32_t *__restrict__ nbo, int32_t *__restrict__ nbi) {
    const int lane = threadIdx.x & 31;
    const int v = it.x;
    const int r = counts ? bold[v] : -1, s = bnew[v];
    const int o0 = g.op[v], kout = g.op[v + 1] - o0;
    const int i0 = g.ip[v], k = kout + (g.ip[v + 1] - i0);
    if (r == s) return;
    const int hi = min(k, (it.y + 1) * kMoveChunk);
    for (int lo = it.y * kMoveChunk; lo < hi; lo += 32 * kItemIn) {
        int nb[kItemIn], tw[kItemIn], t[kItemIn], u[kItemIn];
#pragma unroll
        for (int j = 0; j < kItemIn; ++j) {
            const int idx = lo + j * 32 + lane;
            const bool out = idx < kout;
            const int at = out ? o0 + idx : i0 + idx - kout;
            nb[j] = idx < hi ? (out ? g.oc : g.ic)[at] : -1;
            tw[j] = nbo && idx < hi ? (out ? g.tw_oi : g.tw_io)[at] : 0;
        }
#pragma unroll
        for (int j = 0; j < kItemIn; ++j) {
            t[j] = counts && nb[j] >= 0 ? bold[nb[j]] : 0;
            u[j] = counts && nb[j] >= 0 ? bnew[nb[j]] : 0;
        }
        if (nbo) {
#pragma unroll
            for (int j = 0; j < kItemIn; ++j) {
                // v -> w: in w's in-row; w -> v: in w's out-row
                if (nb[j] >= 0) (lo + j * 32 + lane < kout ? nbi : nbo)[tw[j]] = s | (nb[j] == v ? kNbSelf : 0);
            }
        }
        if (!counts) continue;
#pragma unroll
        for (int j = 0; j < kItemIn; ++j) {
            int leave = -1, enter = -1;  // cells (B * B <= 2^26) the edge leaves and enters
            if (nb[j] >= 0) {
                if (lo + j * 32 + lane < kout) {
                    // out-edge v -> w: leaves (r, t), enters (s, u)
                    leave = r * B + t[j];
                    enter = s * B + u[j];
                } else if (u[j] == t[j]) {
                    // in-edge w -> v from a vertex that stayed (a moved
                    // source applies it through its own out-row)
                    leave = t[j] * B + r;
                    enter = t[j] * B + s;
                }
            }
            warp_cell_add(M, leave, -1);
            warp_cell_add(M, enter, 1);
        }
    }
}

// The same apply step driven by the accepted-move list: an item is one
// kMoveChunk-edge slice of the concatenated (out, in) row of a moved vertex,
// so hubs are spread over many warps and no warp scans unmoved vertices.
// The block-labelled rows (nbo not NULL) follow whatever the plan; the count
// update runs only when the plan chose it.
constexpr int kItemCtas = 8;  // per SM

__global__ void __launch_bounds__(kThreads, kItemCtas) k_delta_items(GraphDev g, const int2 *__restrict__ items,
                                                          const DevCounters *__restrict__ c, int64_t cap,
                                                          const int32_t *__restrict__ bnew,
                                                          const int32_t *__restrict__ bold, int32_t *__restrict__ M,
                                                          int B, const int32_t *__restrict__ flag,
                                                          int32_t *__restrict__ nbo, int32_t *__restrict__ nbi) {
    const bool counts = *flag == 1;
    if (!counts && !nbo) return;
    const int64_t total = (int64_t)(c->items < (unsigned long long)cap ? c->items : (unsigned long long)cap);
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < total; w += nw)
        delta_item(g, items[w], bnew, bold, M, B, counts, nbo, nbi);
}

// block-labelled rows from scratch, both CSRs in their own order (coalesced
// writes): out-entry e (u -> w) gets b[w], in-entry j (w -> u) gets b[w];
// bit 31 marks a self-loop (out-rows: from the edge's source; in-rows: set
// afterwards at the graph's self-loop positions by k_nb_self)
__global__ void k_nb_full(GraphDev g, const int32_t *__restrict__ b, int32_t *__restrict__ nbo,
                          int32_t *__restrict__ nbi) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < g.m; e += stride) {
        const int u = g.esrc[e], w = g.oc[e], x = g.ic[e];
        nbo[e] = b[w] | (u == w ? kNbSelf : 0);
        nbi[e] = b[x];
    }
}

__global__ void k_nb_self(const int32_t *__restrict__ self_in, int64_t n_self, int32_t *__restrict__ nbi) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_self; i += (int64_t)gridDim.x * blockDim.x)
        nbi[self_in[i]] |= kNbSelf;
}

// the entries that name a moved vertex, after a pass: for every item of
// the accepted-move list (a 256-edge slice of moved vertex v's rows), the
// twin of each of v's edges takes v's new label
__global__ void __launch_bounds__(kThreads, kItemCtas) k_nb_items(GraphDev g, const int2 *__restrict__ items,
                                                                  const DevCounters *__restrict__ c, int64_t cap,
                                                                  const int32_t *__restrict__ b,
                                                                  int32_t *__restrict__ nbo, int32_t *__restrict__ nbi) {
    const int64_t total = (int64_t)(c->items < (unsigned long long)cap ? c->items : (unsigned long long)cap);
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < total; w += nw)
        delta_item(g, items[w], b, nullptr, nullptr, 0, false, nbo, nbi);
}

// ---------------------------------------------------------------------------
// The commit of a small dense model in one launch of one cluster: plan, cells
// (update or recount) with the block-labelled rows, prefix rows, degrees, DL,
// the pending labels, and what the host reads, with cluster barriers where
// the separate kernels have launches.  At these sizes each of the nine stream
// operations it replaces is a few microseconds of launch and drain around
// less than one of work.  With k_eval_small, three sweeps at 1000 vertices
// and 8 blocks, their labels set before and read back after, took 209 us
// instead of 526.
// Its eight SMs are few for much work, so its use has three limits (labels set
// from outside and committed, the separate kernels and this one, in us):
//   - blocks, whose prefix rows it builds on 256 warps (2000 vertices, 8000
//     edges, nothing moved): 66 and 51 at B = 256, 71 and 68 at 384, 74 and 77
//     at 512; with a pass before it and its statistics read (3000 vertices,
//     40,000 edges), 91 and 67 at 300, 91 and 82 at 500;
//   - moves: an item costs some 6 ns, an edge end of an update 0.15 ns, an edge
//     of a recount 0.075 ns, and the blocks' rows add up, against the launches
//     it saves; commit_max_load is that budget in items.  A pass's commit also
//     saves the copies that read its statistics back: B = 128, 8000 vertices,
//     130,000 edges, load 4670 57 and 49; 12,000, 170,000, 6540 57 and 57;
//     20,000, 130,000, 6080 57 and 53, 9360 58 and 67; 60,000, 500,000, 6850 59
//     and 63; B = 64: 12,000, 170,000, 6340 57 and 56; B = 256: 5720 57 and 54,
//     7470 58 and 63.  At few blocks the separate kernels wait for one another
//     at the counts, B = 8: 20,000 vertices, 520,000 edges, 9790 142 and 129,
//     12,400 156 and 167; 40,000, 300,000, 10,990 107 and 98, 17,900 120 and
//     133.  Labels set from outside, nothing read, B = 128: 8000, 130,000, 3530
//     76 and 70, 6600 82 and 84; 20,000, 500,000, 2600 80 and 67, 4920 82 and
//     83, 10,600 83 and 110; 65,000, 520,000, 4760 82 and 80, 45,000 91 and 266;
//   - vertices and edges, up to which these were measured.
// Where not every commit of the model is within the load, the kernel looks at
// the moves first and leaves the commit to the separate kernels when there
// are too many (a launch and a wait lost).  It is not asked after a pass with
// (or labels set from outside) more than kCommitTryFactor times the load: from
// one pass to the next the moves rarely fall by more.
constexpr int kCommitThreads = 1024;
constexpr int kCommitCluster = 8;
constexpr int kCommitMaxB = 512, kCommitMaxSetB = 256;  // of a pass, of labels set from outside
constexpr int64_t kCommitMaxEdges = int64_t(1) << 19;
constexpr int64_t kCommitMaxVertices = int64_t(1) << 16;
constexpr unsigned long long kCommitTryFactor = 3;

__host__ __device__ inline unsigned long long commit_max_load(int B) {
    return 6000 + 32000 / (B > 8 ? B : 8);  // (fewer than 8 blocks were not measured)
}

__host__ __device__ inline bool commit_counts_moves(const DevCounters &c, int64_t m) {
    return c.acc_edges * 4ull <= (unsigned long long)m;  // else all edges are counted again
}

__host__ __device__ inline unsigned long long commit_load(const DevCounters &c, int64_t m, int B) {
    return c.items + (commit_counts_moves(c, m) ? c.acc_edges / 40 : (unsigned long long)m / 80) +
           (unsigned long long)B * B / 64;
}

struct SmallCommit {
    GraphDev g;
    const int2 *items;
    int64_t cap_items;
    DevCounters *counters;
    const int32_t *b;  // the new labels
    int32_t *bold;     // the previous ones; takes the new ones at the end
    int32_t *M;
    int B, pstep;
    uint32_t *P, *Pc;
    int32_t *dout, *din, *dsum;
    double *rcp;
    float *rcp32;
    const __int128 *T;  // holds every count (the edges are below its size)
    int32_t *nbo, *nbi;
    double *dl;
    DlPartial *parts;  // one per block of the cluster
    const int32_t *status;
    SweepReadback *host;  // NULL: not asked for
    bool checked;         // the load is looked at first (with host)
};

__global__ void __launch_bounds__(kCommitThreads) k_commit_small(SmallCommit a) {
    __shared__ int diag[kCommitMaxB];
    __shared__ __int128 sfix[kCommitThreads / 32];
    __shared__ double s_model;
    const int B = a.B, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int tid = cluster_rank() * kCommitThreads + threadIdx.x, nt = cluster_size() * kCommitThreads;
    const DevCounters c = *a.counters;
    if (a.checked && commit_load(c, a.g.m, B) > commit_max_load(B)) {
        if (tid == 0) a.host->done = 0;
        return;
    }
    const bool counts = commit_counts_moves(c, a.g.m);
    const int64_t items = (int64_t)(c.items < (unsigned long long)a.cap_items ? c.items : (unsigned long long)a.cap_items);
    // the part of DL that does not need the counts (a chain of FP64
    // logarithms) on a thread of its own
    if (tid == kCommitThreads - 1) s_model = dl_eq2(a.g.m, a.g.n, B, 0.0);
    if (!counts) {
        for (int i = threadIdx.x; i < B; i += kCommitThreads) diag[i] = 0;
        for (int i = tid; i < B * B; i += nt) a.M[i] = 0;
        cluster_sync();
        for (int64_t e = tid; e < a.g.m; e += nt) hist_add(a.M, diag, B, true, a.b[a.g.esrc[e]], a.b[a.g.oc[e]]);
        __syncthreads();
        for (int i = threadIdx.x; i < B; i += kCommitThreads)
            if (diag[i]) atomicAdd(&a.M[(size_t)i * B + i], diag[i]);
    }
    if (counts || a.nbo)
        for (int64_t w = tid >> 5; w < items; w += nt >> 5)
            delta_item(a.g, a.items[w], a.b, a.bold, a.M, B, counts, a.nbo, a.nbi);
    cluster_sync();
    __int128 fix = 0;
    for (int u = tid >> 5; u < B; u += nt >> 5) {
        prefix_block<false>(a.M, B, u, a.P, a.dout, a.din, a.rcp, a.rcp32, a.dsum, a.Pc, a.pstep);
        if (lane == 0) fix -= a.T[a.dout[u]] + a.T[a.din[u]];
    }
    for (int i = tid; i < B * B; i += nt) fix += a.T[__ldcg(&a.M[i])];
    for (int v = tid; v < a.g.n; v += nt) a.bold[v] = a.b[v];
    fix = warp_sum_128(fix);
    if (lane == 0) sfix[wid] = fix;
    __syncthreads();
    if (threadIdx.x == 0) {
        __int128 f = 0;
        for (int q = 0; q < kCommitThreads / 32; ++q) f += sfix[q];
        a.parts[cluster_rank()].fix = f;
    }
    cluster_sync();
    if (tid == 0) {
        __int128 f = 0;
        for (int q = 0; q < cluster_size(); ++q) f += a.parts[q].fix;
        const double before = a.dl[0], after = s_model - fix_to_double(f);
        a.dl[0] = after;
        a.dl[1] = before;
        if (a.host) {
            a.host->c = c;
            a.host->dl[0] = after;
            a.host->dl[1] = before;
            a.host->status = *a.status;
            a.host->done = 1;
        }
        *a.counters = DevCounters{};
    }
}

__global__ void k_relabel(int32_t *__restrict__ b, int32_t *__restrict__ bnew, int n, const int32_t *__restrict__ map) {
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const int x = map[b[v]];
        b[v] = x;
        bnew[v] = x;
    }
}

__global__ void k_vertex_count(const int32_t *__restrict__ b, int n, int32_t *__restrict__ cnt) {
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) atomicAdd(&cnt[b[v]], 1);
}

int grid_for(int64_t work, int per_block, int cap) {
    int64_t g = (work + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

int num_sms() {
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

size_t dense_bytes(int64_t B) {
    const size_t b = (size_t)B, chunks = (b + kColChunk - 1) / kColChunk;
    return 12 * b * b + 128 * b + (B >= kWidePrefixB ? 4 * b * chunks : 0);
}

size_t block_bytes(int64_t B) { return 44 * (size_t)B; }

size_t label_row_bytes(const sbp_graph *g) { return 8 * (size_t)g->m; }

// (dense_bytes and block_bytes say how much this allocates)
int ensure_capacity(sbp_model *m, int32_t B) {
    m->dense = B <= m->p.dense_max_B;
    if (!m->dense) SBP_TRY(ensure_sparse_capacity(m, B));
    const bool need_dense = m->dense && B > m->Bdense;
    if (B <= m->Bcap && !need_dense) return SBP_OK;
    cudaStream_t st = m->stream;
    auto alloc = [&](auto **p, size_t bytes) { return model_alloc((void **)p, bytes, st) == cudaSuccess; };
    if (need_dense) {
        model_free(m->M, st);
        model_free(m->P, st);
        model_free(m->Pc, st);
        model_free(m->colsum, st);
        m->M = nullptr; m->P = nullptr; m->Pc = nullptr; m->colsum = nullptr;
        m->Bdense = 0;
        const size_t BB = (size_t)B * B;
        if (!alloc(&m->M, BB * 4) || !alloc(&m->P, BB * 8) || !alloc(&m->Pc, (size_t)B * 32 * 4) ||
            (B >= kWidePrefixB && !alloc(&m->colsum, (size_t)B * ((B + kColChunk - 1) / kColChunk) * 4))) {
            cudaGetLastError();
            return fail(SBP_ENOMEM, "device allocation failed for a dense blockmodel of B = " + std::to_string(B));
        }
        m->Bdense = B;
    }
    if (B > m->Bcap) {
        void *old[] = {m->dout, m->din, m->rcp, m->rcp32, m->dsum, m->best_s, m->best_d, m->map, m->vcount};
        for (void *p : old) model_free(p, st);
        m->dout = m->din = nullptr; m->rcp = nullptr; m->rcp32 = nullptr; m->dsum = nullptr;
        m->best_s = m->map = m->vcount = nullptr; m->best_d = nullptr;
        m->Bcap = 0;
        const size_t b = (size_t)B;
        if (!alloc(&m->dout, b * 4) || !alloc(&m->din, b * 4) || !alloc(&m->rcp, b * 8) || !alloc(&m->rcp32, b * 4) ||
            !alloc(&m->dsum, b * 4) || !alloc(&m->best_s, b * 4) || !alloc(&m->best_d, b * 8) ||
            !alloc(&m->map, b * 4) || !alloc(&m->vcount, b * 4)) {
            cudaGetLastError();
            return fail(SBP_ENOMEM, "device allocation failed for the block arrays of B = " + std::to_string(B));
        }
        m->Bcap = B;
    }
    return SBP_OK;
}

// cells[r * B + t] = number of edges from block r to block t (all B * B
// cells are written); B <= 16384
int count_cells(sbp_model *m, int32_t *cells) {
    const sbp_graph *g = m->g;
    const int B = m->B;
    SBP_CUDA(cudaMemsetAsync(cells, 0, (size_t)B * B * 4, m->stream));
    if (g->m > 0) {
        const size_t smem = (size_t)B * 4;
        if (smem > 48 * 1024)
            SBP_TRY(ensure_dyn_smem((const void *)k_hist_dense, smem));
        k_hist_dense<<<grid_for((g->m + 3) / 4, kThreads, num_sms() * 8), kThreads, smem, m->stream>>>(g->dev(), m->b,
                                                                                                        cells, B, nullptr);
        SBP_LAUNCHED();
    }
    return SBP_OK;
}

// cells (the counts of the previous assignment m->bnew) brought to the
// counts of m->b: the plan kernel picks, on the device, either the update
// from the moved vertices' rows (few moved edges) or a recount; both give
// the same counts
int update_cells(sbp_model *m, int32_t *cells) {
    const sbp_graph *g = m->g;
    const int B = m->B;
    const int sms = num_sms();
    const int64_t BB = (int64_t)B * B;
    int32_t *flag = m->status + 1;
    k_commit_plan<<<grid_for(BB, kThreads, sms * 8), kThreads, 0, m->stream>>>(m->counters, g->m, flag, cells, BB);
    SBP_LAUNCHED();
    if (g->m > 0) {
        const size_t smem = (size_t)B * 4;
        if (smem > 48 * 1024)
            SBP_TRY(ensure_dyn_smem((const void *)k_hist_dense, smem));
        k_hist_dense<<<grid_for((g->m + 3) / 4, kThreads, sms * 8), kThreads, smem, m->stream>>>(g->dev(), m->b, cells, B,
                                                                                                  flag);
        SBP_LAUNCHED();
        if (m->list_ok && m->items) {
            // the block-labelled rows follow in the same pass
            const bool nb = m->nb_ok && m->nbo;
            k_delta_items<<<sms * kItemCtas, kThreads, 0, m->stream>>>(g->dev(), m->items, m->counters, m->cap_items, m->b,
                                                               m->bnew, cells, B, flag, nb ? m->nbo : nullptr,
                                                               nb ? m->nbi : nullptr);
            SBP_LAUNCHED();
            m->nb_in_commit = nb;
        } else {
            const int64_t n_big = g->n - g->bin[3];
            const int64_t warps = n_big + (g->n + 31) / 32;
            k_delta_dense<<<grid_for(warps * 32, kThreads, 1 << 30), kThreads, 0, m->stream>>>(
                g->dev(), g->order, (int)g->bin[3], (int)n_big, m->b, m->bnew, cells, B, flag);
            SBP_LAUNCHED();
        }
    }
    return SBP_OK;
}

namespace {

int launch_wide_prefix(sbp_model *m, DlPartial *parts, int *np) {
    const int B = m->B;
    const int ub = (B + 31) / 32, chunks = (B + kColChunk - 1) / kColChunk;
    const int rows = std::min(B, num_sms() * 8), fin = (B + kThreads / 32 - 1) / (kThreads / 32);
    static_assert(16384 / (kThreads / 32) + 152 * 8 <= kPartials, "the partials of L");
    uint32_t *sums = m->colsum;
    k_prefix_rows<<<rows, kThreads, 0, m->stream>>>(m->M, B, m->P, m->dout, m->T, m->XT, parts);
    SBP_LAUNCHED();
    k_col_sums<<<dim3(ub, chunks), kThreads, 0, m->stream>>>(m->M, B, sums);
    SBP_LAUNCHED();
    k_prefix_cols<<<dim3(ub, chunks), kThreads, 0, m->stream>>>(m->M, B, sums, m->dout, m->P);
    SBP_LAUNCHED();
    k_wide_finish<<<fin, kThreads, 0, m->stream>>>(m->P, B, m->dout, m->din, m->rcp, m->rcp32, m->dsum, m->Pc,
                                                   (2 * B + 31) / 32, m->T, m->XT, parts + rows);
    SBP_LAUNCHED();
    *np = rows + fin;
    return SBP_OK;
}

// M (dense, or sparse rows), P, degrees, rcp and DL from m->b.  after_pass:
// m->bnew holds the assignment the current M was built from, and the counts
// may be updated from the moves instead of recounted.
int build_blockmodel(sbp_model *m, bool after_pass) {
    const sbp_graph *g = m->g;
    const int B = m->B;
    SBP_TRY(xlogx_table(g->m + 1, &m->T, &m->XT));
    DlPartial *parts = reinterpret_cast<DlPartial *>(m->partials);
    int np = 0;
    if (m->dense) {
        const int64_t BB = (int64_t)B * B;
        if (after_pass)
            SBP_TRY(update_cells(m, m->M));
        else
            SBP_TRY(count_cells(m, m->M));
        if (B >= kWidePrefixB) {
            SBP_TRY(launch_wide_prefix(m, parts, &np));
        } else {
            SBP_TRY(launch_prefix(m));
            np = grid_for(BB > B ? BB : B, kThreads * 4, 1024);  // (of kPartials)
            k_dl_partial<<<np, kThreads, 0, m->stream>>>(m->M, BB, m->dout, m->din, B, m->T, m->XT, parts);
            SBP_LAUNCHED();
        }
        k_dl_final<<<1, kFinalThreads, 0, m->stream>>>(parts, np, g->m, g->n, B, m->dl);
        SBP_LAUNCHED();
    } else {
        bool dl_done = false;
        SBP_TRY(rebuild_sparse(m, after_pass, &dl_done, &np));
        if (!dl_done) {
            k_dl_final<<<1, kFinalThreads, 0, m->stream>>>(parts, np, g->m, g->n, B, m->dl);
            SBP_LAUNCHED();
        }
    }
    SBP_CUDA(cudaMemcpyAsync(m->bnew, m->b, (size_t)g->n * 4, cudaMemcpyDeviceToDevice, m->stream));
    return SBP_OK;
}

}  // namespace

// a rebuild from m->b drops the pending decisions, and with them the
// accepted-move list
int rebuild_blockmodel(sbp_model *m) {
    m->nb_ok = false;
    m->list_ok = true;
    m->decided.clear();
    SBP_CUDA(cudaMemsetAsync(&m->counters->items, 0, sizeof(unsigned long long), m->stream));
    return build_blockmodel(m, false);
}

// P, Pc, degrees and reciprocals of a dense model from its M
int launch_prefix(sbp_model *m) {
    const int B = m->B;
    k_prefix_dense<<<grid_for((int64_t)B * 32, kThreads, 1 << 30), kThreads, 0, m->stream>>>(
        m->M, B, m->P, m->dout, m->din, m->rcp, m->rcp32, m->dsum, m->Pc, (2 * B + 31) / 32);
    SBP_LAUNCHED();
    return SBP_OK;
}

// After a nodal pass (m->b: new labels, m->bnew: the previous ones).  The
// counts (dense M, or the cell counts of a sparse model rebuilt by
// counting) take the incremental update when the plan kernel finds few
// moved edges (decided on the device, no host round trip); the result is
// the same M as a recount.
int commit_blockmodel(sbp_model *m) { return build_blockmodel(m, !m->p.full_rebuild); }

// the small form: a dense model within its limits whose accepted-move list
// holds every change
bool commit_small_ok(const sbp_model *m) {
    return m->dense && !m->p.full_rebuild && m->list_ok && m->items && m->B <= kCommitMaxB &&
           m->g->m <= kCommitMaxEdges && m->g->n <= kCommitMaxVertices;
}

// all vertices moved, all edges counted again
bool commit_small_fits(const sbp_model *m) {
    const sbp_graph *g = m->g;
    return (unsigned long long)(g->n + 2 * g->m / kMoveChunk + g->m / 80 + (int64_t)m->B * m->B / 64) <=
           commit_max_load(m->B);
}

bool commit_small_load_ok(const sbp_model *m, const DevCounters &c) {
    return m->B <= kCommitMaxSetB && commit_load(c, m->g->m, m->B) <= commit_max_load(m->B);
}

bool commit_small_try_next(const sbp_model *m, const DevCounters &c) {
    return commit_load(c, m->g->m, m->B) <= kCommitTryFactor * commit_max_load(m->B);
}

int commit_small(sbp_model *m, SweepReadback *host, bool checked) {
    SBP_TRY(xlogx_table(m->g->m + 1, &m->T, &m->XT));
    const bool nb = m->nb_ok && m->nbo;
    SmallCommit a;
    a.g = m->g->dev();
    a.items = m->items;
    a.cap_items = m->cap_items;
    a.counters = m->counters;
    a.b = m->b;
    a.bold = m->bnew;
    a.M = m->M;
    a.B = m->B;
    a.pstep = (2 * m->B + 31) / 32;
    a.P = m->P;
    a.Pc = m->Pc;
    a.dout = m->dout;
    a.din = m->din;
    a.dsum = m->dsum;
    a.rcp = m->rcp;
    a.rcp32 = m->rcp32;
    a.T = m->T;
    a.nbo = nb ? m->nbo : nullptr;
    a.nbi = nb ? m->nbi : nullptr;
    a.dl = m->dl;
    a.parts = reinterpret_cast<DlPartial *>(m->partials);
    a.status = m->status;
    a.host = host;
    a.checked = checked;
    return launch_cluster(k_commit_small, kCommitCluster, kCommitThreads, 0, m->stream, 1, a);
}

// block-labelled rows from m->b (allocated on first use).  Without the
// memory for them nb_ok stays false and the pass gathers labels instead.
int nb_rows_rebuild(sbp_model *m) {
    const sbp_graph *g = m->g;
    if (!m->nbo) {
        const size_t bytes = (size_t)(g->m > 0 ? g->m : 1) * 4;
        if (model_alloc((void **)&m->nbo, bytes, m->stream) != cudaSuccess ||
            model_alloc((void **)&m->nbi, bytes, m->stream) != cudaSuccess) {
            cudaGetLastError();
            model_free(m->nbo, m->stream);
            model_free(m->nbi, m->stream);
            m->nbo = m->nbi = nullptr;
            return SBP_OK;
        }
    }
    if (g->m > 0) {
        k_nb_full<<<grid_for(g->m, kThreads, num_sms() * 8), kThreads, 0, m->stream>>>(g->dev(), m->b, m->nbo, m->nbi);
        SBP_LAUNCHED();
    }
    if (g->n_self > 0) {
        k_nb_self<<<grid_for(g->n_self, kThreads, num_sms() * 8), kThreads, 0, m->stream>>>(g->self_in, g->n_self,
                                                                                           m->nbi);
        SBP_LAUNCHED();
    }
    m->nb_ok = true;
    return SBP_OK;
}

// after a commit: the block-labelled rows follow the accepted moves, or are
// marked stale when the list does not hold every change
int nb_rows_after_commit(sbp_model *m) {
    if (m->nb_in_commit) {  // updated by the apply step's kernel
        m->nb_in_commit = false;
        return SBP_OK;
    }
    if (!m->nb_ok || !m->nbo) return SBP_OK;
    if (!m->list_ok || !m->items) {
        m->nb_ok = false;
        return SBP_OK;
    }
    k_nb_items<<<num_sms() * kItemCtas, kThreads, 0, m->stream>>>(m->g->dev(), m->items, m->counters, m->cap_items, m->b,
                                                          m->nbo, m->nbi);
    SBP_LAUNCHED();
    return SBP_OK;
}

int launch_relabel(sbp_model *m, const int32_t *map_dev) {
    const int n = (int)m->g->n;
    k_relabel<<<grid_for(n, kThreads, num_sms() * 8), kThreads, 0, m->stream>>>(m->b, m->bnew, n, map_dev);
    SBP_LAUNCHED();
    return SBP_OK;
}

int launch_vertex_count(sbp_model *m) {
    const int n = (int)m->g->n;
    SBP_CUDA(cudaMemsetAsync(m->vcount, 0, (size_t)m->B * 4, m->stream));
    k_vertex_count<<<grid_for(n, kThreads, num_sms() * 8), kThreads, 0, m->stream>>>(m->b, n, m->vcount);
    SBP_LAUNCHED();
    return SBP_OK;
}

}  // namespace sbp
