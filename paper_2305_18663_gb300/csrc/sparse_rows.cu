// sparse_rows.cu -- the sparse rows and columns of M from the assignment, at
// any number of blocks (Section III-A (a)-(b); sparse.cu takes the small ones).
//
// Row r of M is the multiset of the labels at the far ends of the out-edges
// of block r's vertices, column r the same of its in-edges.  The graph's
// rows already group the edges by vertex, so only the vertices have to be
// grouped by block, and every row is then sorted and counted by itself:
//   1. block degrees (k_rows_degrees), then the first slot of every row,
//      column and row table, and the per-block scalars (k_rows_offsets).  A
//      row is given as many slots as it has edges and keeps its nonzeros at
//      their front (rp[r] .. re[r]), so that nothing waits for the nonzeros
//      to be counted;
//   2. every vertex takes a run of slots in its block's row and column
//      (k_rows_slots), and the labels of its edges' far ends are written
//      there (k_rows_labels);
//   3. a row's labels are sorted; its runs of equal labels are the nonzeros,
//      the end of a run is the inclusive prefix of the counts.  Up to 128
//      labels: a warp, a bitonic network in registers (k_rows_small).  Up to
//      512, 4096, 16384: a block of 64, 256, 1024 threads, chunks sorted by
//      its warps and merged in shared memory, or, at few columns, counted
//      (k_rows_mid).  More: a block counts them in windows of columns
//      (k_rows_big).  All fill the row's table and pivots and add its share of
//      L (Eq. 1).
// Rebuilding the rows of a 200k-vertex, 4M-edge graph takes 429 us at
// B = 65,536 (992 for the radix sort of all (row, column) keys, run-length
// encoding, sort by column, table fill and row prefixes that this replaces:
// 55 launches and a read-back), 437 us at 16,384 (938), 285 us at 4096 (467
// from cell counts).  Its 4M labels and their rows, columns and tables are
// some 250 MB of traffic; the row kernels are bound by instruction issue and
// the latency of a row's chain (26 to 44% of the issue slots).  The lines
// between the classes: one class up to 4096 on blocks of 256 threads left
// most of their warps idle on rows of 129 to 512 labels (274 us for both
// classes, 104 + 147 with blocks of 64 for these).
#include "merge_apply.cuh"  // cta_scan
#include "apply.cuh"

#include <algorithm>
#include <climits>

namespace sbp {
namespace {

constexpr int kT = 256;
constexpr int kRowSmall = 128;   // labels of a row one warp sorts
constexpr int kRowHalf = 512;    // ... a block of 64 threads sorts
constexpr int kRowMid = 4096;    // ... a block of 256
constexpr int kRowWide = 16384;  // ... a block of 1024
constexpr int kChunk = 1024;     // blocks (of the model) per thread block of the offsets
constexpr int kRowWindow = 32768;  // columns counted at a time in longer rows
constexpr int kRowBigThreads = 1024;

struct Rows {
    GraphDev g;
    const int32_t *b;
    int32_t B;
    int32_t *dout, *din, *dsum;
    double *rcp;
    float *rcp32;
    uint32_t *rp, *re, *cp, *ce, *hoff;  // row and column begins and ends, table offsets
    uint32_t *rcur, *ccur;               // the next free slot of each row and column
    uint32_t *vo, *vi;                   // a vertex's first slot, less its first edge's position
    int32_t *lo, *li;                    // labels by row, by column
    int32_t *rc, *rv, *cr, *cv;
    uint32_t *rpre, *cpre, *rpc, *cpc;
    int2 *hkv;
    uint32_t *list[4];  // rows (r) and columns (B + r) above kRowSmall, kRowHalf, kRowMid, kRowWide
    uint32_t *count;    // their numbers
    uint32_t *sums;     // [chunks of blocks][kNeeds]
    const __int128 *T;
    int64_t XT;
    DlPartial *parts;
    int32_t *status;
};

// block degrees (zero on entry)
__global__ void __launch_bounds__(kT) k_rows_degrees(Rows a) {
    for (int64_t v = (int64_t)blockIdx.x * kT + threadIdx.x; v < a.g.n; v += (int64_t)gridDim.x * kT) {
        const int r = a.b[v];
        const int ko = a.g.op[v + 1] - a.g.op[v], ki = a.g.ip[v + 1] - a.g.ip[v];
        if (ko) atomicAdd(&a.dout[r], ko);
        if (ki) atomicAdd(&a.din[r], ki);
    }
}

__device__ __forceinline__ uint32_t row_table_slots(uint32_t len, uint32_t B) {
    const uint32_t most = len < B ? len : B;  // distinct columns at most
    return most <= 1 ? 2u : 1u << (32 - __clz((int)(2 * most - 1)));
}

// what block r's row and column need: slots, table slots, places in the lists
struct RowNeeds {
    uint32_t o, i, t, cls[4];
};
constexpr int kNeeds = 7;
__device__ __forceinline__ int row_class(uint32_t len) {
    return len <= kRowSmall ? 0 : len <= kRowHalf ? 1 : len <= kRowMid ? 2 : len <= kRowWide ? 3 : 4;
}
__device__ __forceinline__ RowNeeds row_needs(const Rows &a, int64_t r) {
    RowNeeds x = {0, 0, 0, {0, 0, 0, 0}};
    if (r >= a.B) return x;
    x.o = (uint32_t)a.dout[r];
    x.i = (uint32_t)a.din[r];
    x.t = row_table_slots(x.o, (uint32_t)a.B);
    const int co = row_class(x.o), ci = row_class(x.i);
#pragma unroll
    for (int c = 0; c < 4; ++c) x.cls[c] = (co == c + 1) + (ci == c + 1);
    return x;
}

// sums of the needs of kChunk blocks
__global__ void __launch_bounds__(kChunk) k_rows_sums(Rows a) {
    __shared__ uint32_t sh[kNeeds];
    if (threadIdx.x < kNeeds) sh[threadIdx.x] = 0;
    __syncthreads();
    const RowNeeds x = row_needs(a, (int64_t)blockIdx.x * kChunk + threadIdx.x);
    const uint32_t v[kNeeds] = {x.o, x.i, x.t, x.cls[0], x.cls[1], x.cls[2], x.cls[3]};
#pragma unroll
    for (int q = 0; q < kNeeds; ++q) {
        const uint32_t t = __reduce_add_sync(0xffffffffu, v[q]);
        if ((threadIdx.x & 31) == 0 && t) atomicAdd(&sh[q], t);
    }
    __syncthreads();
    if (threadIdx.x < kNeeds) a.sums[(size_t)blockIdx.x * kNeeds + threadIdx.x] = sh[threadIdx.x];
}

// begins of the rows, columns and tables, the lists in order, the per-block
// scalars; each thread block adds up the sums of the ones before it
__global__ void __launch_bounds__(kChunk) k_rows_offsets(Rows a) {
    __shared__ uint32_t scan[33], base[kNeeds];
    if (threadIdx.x < kNeeds) base[threadIdx.x] = 0;
    __syncthreads();
    uint32_t before[kNeeds] = {};
    for (uint32_t c = threadIdx.x; c < blockIdx.x; c += kChunk)
#pragma unroll
        for (int q = 0; q < kNeeds; ++q) before[q] += a.sums[(size_t)c * kNeeds + q];
#pragma unroll
    for (int q = 0; q < kNeeds; ++q) {
        const uint32_t t = __reduce_add_sync(0xffffffffu, before[q]);
        if ((threadIdx.x & 31) == 0 && t) atomicAdd(&base[q], t);
    }
    __syncthreads();
    const int64_t r = (int64_t)blockIdx.x * kChunk + threadIdx.x;
    const RowNeeds x = row_needs(a, r);
    uint32_t all;
    const uint32_t so = base[0] + cta_scan(x.o, scan, all), si = base[1] + cta_scan(x.i, scan, all);
    const uint32_t st = base[2] + cta_scan(x.t, scan, all);
    uint32_t at[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        at[c] = base[3 + c] + cta_scan(x.cls[c], scan, all);
        if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) a.count[c] = base[3 + c] + all;
    }
    if (r >= a.B) return;
    a.rp[r] = a.rcur[r] = so;
    a.cp[r] = a.ccur[r] = si;
    a.hoff[r] = st;
    if (r == a.B - 1) a.hoff[a.B] = st + x.t;
#pragma unroll
    for (int col = 0; col < 2; ++col) {
        const int k = row_class(col ? x.i : x.o);
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (k == c + 1) a.list[c][at[c]++] = col ? (uint32_t)a.B + (uint32_t)r : (uint32_t)r;
    }
    const int64_t d = (int64_t)x.o + x.i;
    a.dsum[r] = (int32_t)d;
    a.rcp[r] = 1.0 / ((double)d + (double)a.B);
    a.rcp32[r] = 1.0f / ((float)d + (float)a.B);
}

__global__ void __launch_bounds__(kT) k_rows_slots(Rows a) {
    for (int64_t v = (int64_t)blockIdx.x * kT + threadIdx.x; v < a.g.n; v += (int64_t)gridDim.x * kT) {
        const int r = a.b[v];
        const int o0 = a.g.op[v], ko = a.g.op[v + 1] - o0, i0 = a.g.ip[v], ki = a.g.ip[v + 1] - i0;
        // (less the first edge's position, modulo 2^32: an edge adds its own)
        if (ko) a.vo[v] = atomicAdd(&a.rcur[r], (uint32_t)ko) - (uint32_t)o0;
        if (ki) a.vi[v] = atomicAdd(&a.ccur[r], (uint32_t)ki) - (uint32_t)i0;
    }
}

// the far-end labels of a CSR's entries, each in its row's slots
__global__ void __launch_bounds__(kT) k_rows_labels(const int32_t *__restrict__ row, const int32_t *__restrict__ far,
                                                    const uint32_t *__restrict__ slot, const int32_t *__restrict__ b,
                                                    int64_t m, int32_t *__restrict__ lab) {
    const int64_t stride = (int64_t)gridDim.x * kT;
    for (int64_t e0 = (int64_t)blockIdx.x * kT + threadIdx.x; e0 < m; e0 += 4 * stride) {
        int v[4], w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t e = e0 + u * stride;
            v[u] = e < m ? row[e] : 0;
            w[u] = e < m ? far[e] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t e = e0 + u * stride;
            if (e < m) lab[slot[v[u]] + (uint32_t)e] = b[w[u]];
        }
    }
}

// where a row's or a column's nonzeros go
struct RowOut {
    int32_t *idx, *val;
    uint32_t *pre, *piv;
    uint32_t first, len;  // first slot, labels
    const int32_t *lab;
    int32_t r;
    bool col;
};

__device__ __forceinline__ RowOut row_out(const Rows &a, uint32_t id) {
    RowOut o;
    o.col = id >= (uint32_t)a.B;
    o.r = (int32_t)(o.col ? id - (uint32_t)a.B : id);
    o.first = (o.col ? a.cp : a.rp)[o.r];
    o.len = (uint32_t)(o.col ? a.din : a.dout)[o.r];
    o.lab = (o.col ? a.li : a.lo) + o.first;
    o.idx = (o.col ? a.cr : a.rc) + o.first;
    o.val = (o.col ? a.cv : a.rv) + o.first;
    o.pre = (o.col ? a.cpre : a.rpre) + o.first;
    o.piv = (o.col ? a.cpc : a.rpc) + (size_t)o.r * 32;
    return o;
}

// pivot i of a row of D nonzeros whose inclusive prefixes pre(q) gives (the
// layout pivot_upper reads): the end of its i-th segment of ceil(D / 32)
template <class Pre>
__device__ __forceinline__ uint32_t row_pivot(uint32_t i, uint32_t D, Pre pre) {
    const uint32_t step = (D + 31) / 32;
    if (i * step >= D) return 0xffffffffu;
    const uint32_t end = (i + 1) * step < D ? (i + 1) * step : D;
    return pre(end - 1);
}

__device__ __forceinline__ bool row_table_put(int2 *tab, uint32_t cap, int key, int val) {
    uint32_t h = sparse_hash(key) & (cap - 1);
    for (uint32_t t = 0; t < cap; ++t) {
        if (atomicCAS(&tab[h].x, -1, key) == -1) {
            tab[h].y = val;
            return true;
        }
        h = (h + 1) & (cap - 1);
    }
    return false;
}

// a block's share of L into its partial
__device__ void row_partial(DlPartial *part, __int128 fix, double fb) {
    __shared__ __int128 sfix[32];
    __shared__ double sfb[32];
    fix = warp_sum_128(fix);
    fb = warp_sum(fb);
    if ((threadIdx.x & 31) == 0) {
        sfix[threadIdx.x >> 5] = fix;
        sfb[threadIdx.x >> 5] = fb;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < (int)(blockDim.x >> 5); ++q) {
            fix += sfix[q];
            fb += sfb[q];
        }
        part->fix = fix;
        part->fb = fb;
    }
}

// ascending sort of 32 K keys over a warp, lane l holding keys l K .. l K + K - 1
template <int K>
__device__ __forceinline__ void warp_sort(int (&x)[4]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32 * K; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j < K) {
#pragma unroll
                for (int s = 0; s < K; ++s) {
                    if ((s & j) == 0) {
                        const bool up = ((lane * K + s) & k) == 0;
                        const int p = x[s], q = x[s | j];
                        x[s] = up ? min(p, q) : max(p, q);
                        x[s | j] = up ? max(p, q) : min(p, q);
                    }
                }
            } else {
#pragma unroll
                for (int s = 0; s < K; ++s) {
                    const int i = lane * K + s;
                    const int other = __shfl_xor_sync(0xffffffffu, x[s], j / K);
                    const bool keep_min = ((i & k) == 0) == ((i & j) == 0);
                    x[s] = keep_min ? min(x[s], other) : max(x[s], other);
                }
            }
        }
    }
}

struct SmallRow {
    int key[kRowSmall];
    uint32_t start[kRowSmall + 1];
    int2 tab[2 * kRowSmall];
};

template <int K>
__device__ __forceinline__ uint32_t sort_small(const RowOut &o, SmallRow &w) {
    const int lane = threadIdx.x & 31;
    int x[4];
#pragma unroll
    for (int s = 0; s < K; ++s) {
        const uint32_t i = (uint32_t)(s * 32 + lane);  // (any order: it is sorted next)
        x[s] = i < o.len ? o.lab[i] : INT_MAX;
    }
    warp_sort<K>(x);
    const int prev = __shfl_up_sync(0xffffffffu, x[K - 1], 1);
    uint32_t heads = 0, n = 0;
#pragma unroll
    for (int s = 0; s < K; ++s) {
        const uint32_t i = (uint32_t)(lane * K + s);
        const int before = s > 0 ? x[s > 0 ? s - 1 : 0] : prev;
        const bool h = i < o.len && (i == 0 || x[s] != before);
        heads |= (uint32_t)h << s;
        n += h;
    }
    uint32_t rank = warp_incl_scan_u32(n);
    const uint32_t D = __shfl_sync(0xffffffffu, rank, 31);
    rank -= n;
#pragma unroll
    for (int s = 0; s < K; ++s) {
        if ((heads >> s) & 1u) {
            w.start[rank] = (uint32_t)(lane * K + s);
            w.key[rank] = x[s];
            ++rank;
        }
    }
    if (lane == 0) w.start[D] = o.len;
    __syncwarp();
    return D;
}

// a warp per row (tasks [0, B)) or column ([B, 2B)) of at most kRowSmall labels
__global__ void __launch_bounds__(kT) k_rows_small(Rows a) {
    __shared__ SmallRow sw[kT / 32];
    SmallRow &w = sw[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    __int128 fix = 0;
    double fb = 0.0;
    const int64_t nw = ((int64_t)gridDim.x * kT) >> 5;
    for (int64_t id = ((int64_t)blockIdx.x * kT + threadIdx.x) >> 5; id < 2 * (int64_t)a.B; id += nw) {
        const RowOut o = row_out(a, (uint32_t)id);
        if (lane == 0) add_xlogx(a.T, a.XT, o.len, -1, fix, fb);  // the block degree
        if (o.len > kRowSmall) continue;
        const uint32_t off = o.col ? 0u : a.hoff[o.r], cap = o.col ? 0u : a.hoff[o.r + 1] - off;
        for (uint32_t i = lane; i < cap; i += 32) w.tab[i] = make_int2(-1, 0);
        __syncwarp();
        const uint32_t D = o.len == 0 ? 0u
                           : o.len <= 32 ? sort_small<1>(o, w)
                           : o.len <= 64 ? sort_small<2>(o, w)
                                         : sort_small<4>(o, w);
        for (uint32_t q = lane; q < D; q += 32) {
            const int key = w.key[q];
            const uint32_t pre = w.start[q + 1];
            const int val = (int)(pre - w.start[q]);
            o.idx[q] = key;
            o.val[q] = val;
            o.pre[q] = pre;
            if (!o.col) {
                add_xlogx(a.T, a.XT, val, 1, fix, fb);
                if (!row_table_put(w.tab, cap, key, val)) record_status(a.status, SBP_EHASHFULL);
            }
        }
        if (D > 32)  // shorter ones are searched without pivots
            o.piv[lane] = row_pivot((uint32_t)lane, D, [&](uint32_t q) { return w.start[q + 1]; });
        if (lane == 0) (o.col ? a.ce : a.re)[o.r] = o.first + D;
        __syncwarp();
        for (uint32_t i = lane; i < cap; i += 32) a.hkv[off + i] = w.tab[i];
        __syncwarp();
    }
    row_partial(a.parts + blockIdx.x, fix, fb);
}

// a row's table in global memory, cleared and filled by one block from its
// nonzeros (which it wrote before)
__device__ void row_table_global(const Rows &a, const RowOut &o, uint32_t D) {
    if (o.col) return;
    const uint32_t off = a.hoff[o.r], cap = a.hoff[o.r + 1] - off;
    for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x) a.hkv[off + i] = make_int2(-1, 0);
    __syncthreads();
    for (uint32_t q = threadIdx.x; q < D; q += blockDim.x)
        if (!row_table_put(a.hkv + off, cap, o.idx[q], o.val[q])) record_status(a.status, SBP_EHASHFULL);
}

// Sorts n labels (at most CAP) into key: every warp sorts chunks of 128 in
// registers, then runs are merged in pairs, each label finding its place by a
// binary search in the other run.  Returns the buffer it ended in.
template <int THREADS>
__device__ int *sort_labels(const int32_t *__restrict__ lab, int n, int *key, int *tmp) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int P = (n + 127) / 128 * 128;
    for (int c = wid * 128; c < P; c += THREADS * 4) {
        int x[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const int i = c + s * 32 + lane;
            x[s] = i < n ? lab[i] : INT_MAX;
        }
        warp_sort<4>(x);
        *reinterpret_cast<int4 *>(key + c + lane * 4) = make_int4(x[0], x[1], x[2], x[3]);
    }
    __syncthreads();
    for (int width = 128; width < P; width <<= 1) {
        for (int i = threadIdx.x; i < P; i += THREADS) {
            const int x = key[i];
            const int run = i / width * width, pair = i / (2 * width) * (2 * width);
            const bool left = run == pair;
            const int other = left ? pair + width : pair;
            int lo = other, len = other < P ? (P - other < width ? P - other : width) : 0;
            while (len > 0) {  // equal labels: the left run's first
                const int half = len >> 1, y = key[lo + half];
                if (left ? y < x : y <= x) {
                    lo += half + 1;
                    len -= half + 1;
                } else {
                    len = half;
                }
            }
            tmp[pair + (i - run) + (lo - other)] = x;
        }
        __syncthreads();
        int *t = key;
        key = tmp;
        tmp = t;
    }
    return key;
}

// a block per listed row of up to CAP labels
template <int THREADS, int CAP>
__global__ void __launch_bounds__(THREADS) k_rows_mid(Rows a, const uint32_t *__restrict__ list,
                                                      const uint32_t *__restrict__ n_list) {
    extern __shared__ __align__(16) int msm[];
    __shared__ uint32_t scan[33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __int128 fix = 0;
    double fb = 0.0;
    const uint32_t count = *n_list;
    for (uint32_t t = blockIdx.x; t < count; t += gridDim.x) {
        const RowOut o = row_out(a, list[t]);
        uint32_t D;
        if (a.B <= 2 * CAP && (uint32_t)a.B <= 8 * o.len) {
            // few columns: counted, and the nonzeros taken in order
            for (int i = threadIdx.x; i < a.B; i += THREADS) msm[i] = 0;
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < o.len; i += THREADS) atomicAdd(&msm[o.lab[i]], 1);
            __syncthreads();
            const int per = (a.B + THREADS - 1) / THREADS * 32, lo = wid * per, hi = lo + per < a.B ? lo + per : a.B;
            uint32_t nz = 0, sum = 0;
            for (int i0 = lo; i0 < hi; i0 += 32) {
                const int v = i0 + lane < hi ? msm[i0 + lane] : 0;
                nz += v != 0;
                sum += (uint32_t)v;
            }
            uint32_t all;
            uint32_t q = __shfl_sync(0xffffffffu, cta_scan(nz, scan, D), 0);
            uint32_t p = __shfl_sync(0xffffffffu, cta_scan(sum, scan, all), 0);
            for (int i0 = lo; i0 < hi; i0 += 32) {
                const int v = i0 + lane < hi ? msm[i0 + lane] : 0;
                const unsigned nzm = __ballot_sync(0xffffffffu, v != 0);
                const uint32_t incl = warp_incl_scan_u32((uint32_t)v);
                if (v != 0) {
                    const uint32_t at = q + __popc(nzm & ((1u << lane) - 1u));
                    o.idx[at] = i0 + lane;
                    o.val[at] = v;
                    o.pre[at] = p + incl;
                    if (!o.col) add_xlogx(a.T, a.XT, v, 1, fix, fb);
                }
                q += __popc(nzm);
                p += __shfl_sync(0xffffffffu, incl, 31);
            }
        } else {
            int *key = sort_labels<THREADS>(o.lab, (int)o.len, msm, msm + CAP);
            uint32_t *start = reinterpret_cast<uint32_t *>(key == msm ? msm + CAP : msm);
            // runs of equal labels: thread t looks at labels [per t, per (t + 1))
            const int n = (int)o.len, per = (n + THREADS - 1) / THREADS;
            const int lo = min(n, (int)threadIdx.x * per), hi = min(n, lo + per);
            uint32_t heads = 0;
            for (int i = lo; i < hi; ++i) heads += i == 0 || key[i] != key[i - 1];
            uint32_t rank = cta_scan(heads, scan, D);
            for (int i = lo; i < hi; ++i)
                if (i == 0 || key[i] != key[i - 1]) start[rank++] = (uint32_t)i;
            __syncthreads();
            for (uint32_t q = threadIdx.x; q < D; q += THREADS) {
                const uint32_t s = start[q], pre = q + 1 < D ? start[q + 1] : o.len;
                o.idx[q] = key[s];
                o.val[q] = (int)(pre - s);
                o.pre[q] = pre;
                if (!o.col) add_xlogx(a.T, a.XT, pre - s, 1, fix, fb);
            }
        }
        __syncthreads();
        if (threadIdx.x < 32) o.piv[threadIdx.x] = row_pivot(threadIdx.x, D, [&](uint32_t q) { return o.pre[q]; });
        if (threadIdx.x == 0) (o.col ? a.ce : a.re)[o.r] = o.first + D;
        row_table_global(a, o, D);
        __syncthreads();
    }
    row_partial(a.parts + blockIdx.x, fix, fb);
}

// a block per listed row of more than kRowWide labels: counted in windows of
// kRowWindow columns, whose nonzeros are written in order
__global__ void __launch_bounds__(kRowBigThreads) k_rows_big(Rows a) {
    extern __shared__ int cnt[];
    __shared__ uint32_t scan[33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __int128 fix = 0;
    double fb = 0.0;
    const uint32_t count = a.count[3];
    for (uint32_t t = blockIdx.x; t < count; t += gridDim.x) {
        const RowOut o = row_out(a, a.list[3][t]);
        uint32_t D = 0, sum = 0;  // nonzeros and labels of the windows done
        for (int64_t w0 = 0; w0 < a.B; w0 += kRowWindow) {
            const int width = (int)(a.B - w0 < kRowWindow ? a.B - w0 : kRowWindow);
            for (int i = threadIdx.x; i < width; i += kRowBigThreads) cnt[i] = 0;
            __syncthreads();
            for (uint32_t i0 = 0; i0 < o.len; i0 += 8 * kRowBigThreads) {
                int x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const uint32_t i = i0 + u * kRowBigThreads + threadIdx.x;
                    x[u] = i < o.len ? o.lab[i] - (int)w0 : -1;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    // lanes on the first one's column (the diagonal, mostly) add together
                    const int key = x[u] >= 0 && x[u] < width ? x[u] : -1;
                    const unsigned act = __ballot_sync(0xffffffffu, key >= 0);
                    if (!act) continue;
                    const int lead = __ffs(act) - 1, k0 = __shfl_sync(0xffffffffu, key, lead);
                    const unsigned same = __ballot_sync(0xffffffffu, key == k0);
                    if (lane == lead) atomicAdd(&cnt[k0], __popc(same));
                    else if (key >= 0 && key != k0) atomicAdd(&cnt[key], 1);
                }
            }
            __syncthreads();
            // warp w takes columns [per w, per (w + 1)): its nonzeros and their sum
            const int per = (width + kRowBigThreads - 1) / kRowBigThreads * 32;
            const int lo = wid * per, hi = lo + per < width ? lo + per : width;
            uint32_t nz = 0, s = 0;
            for (int i0 = lo; i0 < hi; i0 += 32) {
                const int v = i0 + lane < hi ? cnt[i0 + lane] : 0;
                nz += v != 0;
                s += (uint32_t)v;
            }
            uint32_t nz_all, s_all;
            uint32_t q = cta_scan(nz, scan, nz_all), p = cta_scan(s, scan, s_all);
            q = D + __shfl_sync(0xffffffffu, q, 0);
            p = sum + __shfl_sync(0xffffffffu, p, 0);
            for (int i0 = lo; i0 < hi; i0 += 32) {
                const int v = i0 + lane < hi ? cnt[i0 + lane] : 0;
                const unsigned m = __ballot_sync(0xffffffffu, v != 0);
                const uint32_t incl = warp_incl_scan_u32((uint32_t)v);
                if (v != 0) {
                    const uint32_t at = q + __popc(m & ((1u << lane) - 1u));
                    o.idx[at] = (int)w0 + i0 + lane;
                    o.val[at] = v;
                    o.pre[at] = p + incl;
                    if (!o.col) add_xlogx(a.T, a.XT, v, 1, fix, fb);
                }
                q += __popc(m);
                p += __shfl_sync(0xffffffffu, incl, 31);
            }
            D += nz_all;
            sum += s_all;
            __syncthreads();
        }
        if (threadIdx.x < 32) o.piv[threadIdx.x] = row_pivot(threadIdx.x, D, [&](uint32_t q) { return o.pre[q]; });
        if (threadIdx.x == 0) (o.col ? a.ce : a.re)[o.r] = o.first + D;
        row_table_global(a, o, D);
        __syncthreads();
    }
    row_partial(a.parts + blockIdx.x, fix, fb);
}

// a warp per row: its nonzeros to where they lie without slack
__global__ void __launch_bounds__(kT) k_rows_pack(const uint32_t *__restrict__ rp, const uint32_t *__restrict__ re,
                                                  const uint32_t *__restrict__ first, int B,
                                                  const int32_t *__restrict__ rc, const int32_t *__restrict__ rv,
                                                  int32_t *__restrict__ rc_out, int32_t *__restrict__ rv_out) {
    const int64_t nw = ((int64_t)gridDim.x * kT) >> 5;
    for (int64_t r = ((int64_t)blockIdx.x * kT + threadIdx.x) >> 5; r < B; r += nw) {
        const uint32_t from = rp[r], len = re[r] - from, to = first[r];
#pragma unroll 4
        for (uint32_t i = threadIdx.x & 31; i < len; i += 32) {
            rc_out[to + i] = rc[from + i];
            rv_out[to + i] = rv[from + i];
        }
    }
}

int row_grid(int64_t work, int per_block, int cap) {
    const int64_t g = (work + per_block - 1) / per_block;
    return (int)(g < 1 ? 1 : g > cap ? cap : g);
}

// thread blocks of the row kernels at most: each leaves a partial of L
constexpr int kSms = 152, kG1 = kSms * 8, kG2 = kSms * 12, kG3 = kSms * 4, kG4 = kSms;
static_assert(kG1 + kG2 + kG3 + 2 * kG4 <= kPartials, "the partials of L");

int launch_row_kernels(sbp_model *m, Rows a, const cudaStream_t st[3], int *n_parts) {
    const sbp_graph *g = m->g;
    const int B = m->B;
    // (no more rows above a size than the edges, and the blocks, allow)
    auto rows_above = [&](int64_t len) { return std::min<int64_t>(2 * (int64_t)B, 2 * g->m / len); };
    int parts = 0;
    auto sorted_rows = [&](auto kern, int c, int above, int cap, int threads, int most, cudaStream_t on) -> int {
        const size_t smem = (size_t)2 * cap * 4;
        SBP_TRY(ensure_dyn_smem((const void *)kern, smem));
        const int gr = row_grid(rows_above(above), 1, most);
        kern<<<gr, threads, smem, on>>>(a, a.list[c], a.count + c);
        SBP_LAUNCHED();
        a.parts += gr;
        parts += gr;
        return SBP_OK;
    };
    const int g5 = row_grid(rows_above(kRowWide), 1, kG4);
    const size_t big_smem = (size_t)std::min(B, kRowWindow) * 4;
    SBP_TRY(ensure_dyn_smem((const void *)k_rows_big, big_smem));
    k_rows_big<<<g5, kRowBigThreads, big_smem, st[2]>>>(a);
    SBP_LAUNCHED();
    a.parts += g5;
    parts += g5;
    SBP_TRY(sorted_rows(k_rows_mid<1024, kRowWide>, 2, kRowMid, kRowWide, 1024, kG4, st[2]));
    SBP_TRY(sorted_rows(k_rows_mid<256, kRowMid>, 1, kRowHalf, kRowMid, 256, kG3, st[1]));
    SBP_TRY(sorted_rows(k_rows_mid<64, kRowHalf>, 0, kRowSmall, kRowHalf, 64, kG2, st[2]));
    const int g1 = row_grid(2 * (int64_t)B, kT / 32, kG1);
    k_rows_small<<<g1, kT, 0, st[0]>>>(a);
    SBP_LAUNCHED();
    *n_parts = parts + g1;
    return SBP_OK;
}

}  // namespace

// Rows and columns of M, the block degrees and scalars, and the partials of L
// (*n_parts of them, for the caller's reduction) from m->b.
int build_sparse_rows(sbp_model *m, int *n_parts) {
    const sbp_graph *g = m->g;
    sbp_model::Sparse &S = m->sp;
    cudaStream_t st = m->stream;
    Rows a;
    a.g = g->dev();
    a.b = m->b;
    a.B = m->B;
    a.dout = m->dout;
    a.din = m->din;
    a.dsum = m->dsum;
    a.rcp = m->rcp;
    a.rcp32 = m->rcp32;
    a.rp = S.rp;
    a.re = S.re;
    a.cp = S.cp;
    a.ce = S.ce;
    a.hoff = S.hoff;
    a.rcur = S.rcur;
    a.ccur = S.ccur;
    a.vo = S.vo;
    a.vi = S.vi;
    a.lo = S.lo;
    a.li = S.li;
    a.rc = S.rc;
    a.rv = S.rv;
    a.cr = S.cr;
    a.cv = S.cv;
    a.rpre = S.rpre;
    a.cpre = S.cpre;
    a.rpc = S.rpc;
    a.cpc = S.cpc;
    a.hkv = S.hkv;
    for (int c = 0; c < 4; ++c) a.list[c] = S.lists + 2 * c * (int64_t)S.cap_b;
    a.sums = S.lists + 8 * (int64_t)S.cap_b;
    a.count = S.scratch;
    a.T = m->T;
    a.XT = m->XT;
    a.parts = reinterpret_cast<DlPartial *>(m->partials);
    a.status = m->status;
    const int B = m->B;
    SBP_CUDA(cudaMemsetAsync(m->dout, 0, (size_t)B * 4, st));
    SBP_CUDA(cudaMemsetAsync(m->din, 0, (size_t)B * 4, st));
    k_rows_degrees<<<row_grid(g->n, kT, kSms * 8), kT, 0, st>>>(a);
    SBP_LAUNCHED();
    const int chunks = (int)(((int64_t)B + kChunk - 1) / kChunk);
    k_rows_sums<<<chunks, kChunk, 0, st>>>(a);
    SBP_LAUNCHED();
    k_rows_offsets<<<chunks, kChunk, 0, st>>>(a);
    SBP_LAUNCHED();
    if (g->m > 0) {
        k_rows_slots<<<row_grid(g->n, kT, kSms * 8), kT, 0, st>>>(a);
        SBP_LAUNCHED();
        const int ge = row_grid(g->m, kT * 4, kSms * 8);
        k_rows_labels<<<ge, kT, 0, st>>>(g->esrc, g->oc, S.vo, m->b, g->m, S.lo);
        SBP_LAUNCHED();
        k_rows_labels<<<ge, kT, 0, st>>>(g->idst, g->ic, S.vi, m->b, g->m, S.li);
        SBP_LAUNCHED();
    }
    // the classes' kernels write different rows
    cudaStream_t side[3];
    SBP_TRY(fork_side(m, side));
    const int rc = launch_row_kernels(m, a, side, n_parts);
    const int rj = join_side(m);  // joined on every path
    if (rc != SBP_OK) return rc;
    if (rj != SBP_OK) return rj;
    S.slack = true;
    return SBP_OK;
}

// (the labels and the slot cursors of the build are done with after it)
int pack_sparse_rows(const sbp_model *m, const uint32_t *first, const int32_t **rc, const int32_t **rv) {
    const sbp_model::Sparse &S = m->sp;
    SBP_CUDA(cudaMemcpyAsync(S.rcur, first, (size_t)m->B * 4, cudaMemcpyHostToDevice, m->stream));
    k_rows_pack<<<row_grid(m->B, kT / 32, kSms * 8), kT, 0, m->stream>>>(S.rp, S.re, S.rcur, m->B, S.rc, S.rv, S.lo, S.li);
    SBP_LAUNCHED();
    *rc = S.lo;
    *rv = S.li;
    return SBP_OK;
}

}  // namespace sbp
