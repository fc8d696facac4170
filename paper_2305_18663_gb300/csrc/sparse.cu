// sparse.cu -- the blockmodel as sparse rows (B > dense_max_B).
//
// Section III-A (a)-(b): M held as per-row hashed sparse rows plus a stored
// transpose:
//   - CSR: the nonzeros of every row in ascending column with the inclusive
//     prefix of their counts (the proposal CDF over the row); CSC the same by
//     column;
//   - per-row open-addressing tables (capacity a power of two at least twice
//     the row's length; each slot holds the key and the count, so a probe is
//     one 8-byte load) for M[r][c] lookups;
//   - 32 pivots of every row's and column's prefix;
//   - the block degrees and scalars, and DL.
// Up to kSmallRowsB blocks they are made from the B x B cell counts, which a
// commit can update from the moves (below); at more blocks from the graph's
// rows (sparse_rows.cu).
#include <algorithm>

#include "apply.cuh"

namespace sbp {

namespace {

constexpr int kT = 256;

// Small B (at most kSmallRowsB blocks): the rebuild from the cell counts in
// four kernels with no host round trip -- CSR (offsets, columns, counts,
// in-row prefixes, dout), CSC the same by column (rows ascending), the
// per-row hash tables, the per-block scalars and DL (Eq. 2, exact fixed-point
// sums, the same integer L as the general path).
constexpr int kSmallRowsB = 1024;
constexpr int kSmallThreads = 1024;

__device__ uint32_t cta_excl_scan_1024(uint32_t v, uint32_t *sh, uint32_t *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        const uint32_t t = sh[lane];
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
    *total = sh[32];
    __syncthreads();
    return r;
}

// (1) row and column lengths: a warp per row (warps [0, B)) or per column
// (warps [B, 2B))
__global__ void k_small_lengths(const int32_t *__restrict__ cells, int B, uint32_t *__restrict__ rlen,
                                uint32_t *__restrict__ clen) {
    const int lane = threadIdx.x & 31;
    const int w = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (w >= 2 * B) return;
    const bool col = w >= B;
    const int i = col ? w - B : w;
    uint32_t c = 0;
    for (int j0 = 0; j0 < B; j0 += 32 * 8) {
        int32_t x[8];  // eight chunks of the row (or column) in flight
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = j0 + 32 * q + lane;
            x[q] = j < B ? (col ? cells[j * B + i] : cells[i * B + j]) : 0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) c += (uint32_t)__popc(__ballot_sync(0xffffffffu, x[q] != 0));
    }
    if (lane == 0) (col ? clen : rlen)[i] = c;
}

// (2) one CTA: offsets of the rows, the columns and the row tables
__global__ void __launch_bounds__(kSmallThreads) k_small_offsets(const uint32_t *__restrict__ rlen,
                                                                 const uint32_t *__restrict__ clen, int B,
                                                                 uint32_t *__restrict__ rp, uint32_t *__restrict__ cp,
                                                                 uint32_t *__restrict__ hoff) {
    __shared__ uint32_t sh[33];
    const int tid = threadIdx.x;
    uint32_t total;
    const uint32_t lr = tid < B ? rlen[tid] : 0u;
    uint32_t ex = cta_excl_scan_1024(lr, sh, &total);
    if (tid < B) rp[tid] = ex;
    if (tid == 0) rp[B] = total;
    ex = cta_excl_scan_1024(tid < B ? clen[tid] : 0u, sh, &total);
    if (tid < B) cp[tid] = ex;
    if (tid == 0) cp[B] = total;
    uint32_t cap = 0;
    if (tid < B) {
        cap = 2;
        while (cap < 2 * lr) cap <<= 1;
    }
    ex = cta_excl_scan_1024(cap, sh, &total);
    if (tid < B) hoff[tid] = ex;
    if (tid == 0) hoff[B] = total;
}

// (3) a warp per row (warps [0, B)): CSR entries, in-row prefixes, dout,
// the row's hash table (cleared, then filled by the same warp); a warp per
// column (warps [B, 2B)): CSC entries, prefixes, din.  Per warp, its share
// of L (Eq. 1): + x ln x of the row's counts, - dout ln dout or
// - din ln din, in fixed point.
__global__ void k_small_fill(const int32_t *__restrict__ cells, int B, const uint32_t *__restrict__ rp,
                             const uint32_t *__restrict__ cp, const uint32_t *__restrict__ hoff,
                             int32_t *__restrict__ rc, int32_t *__restrict__ rv, uint32_t *__restrict__ rpre,
                             int32_t *__restrict__ cr, int32_t *__restrict__ cv,
                             uint32_t *__restrict__ cpre, int2 *__restrict__ hkv,
                             int32_t *__restrict__ dout, int32_t *__restrict__ din, const __int128 *__restrict__ T,
                             int64_t XT, __int128 *__restrict__ lpart, double *__restrict__ lfb,
                             int32_t *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int w = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (w >= 2 * B) return;
    const bool col = w >= B;
    const int i = col ? w - B : w;
    __int128 f = 0;
    double fb = 0.0;  // counts beyond the table, in FP64
    uint32_t p = col ? cp[i] : rp[i], carry = 0;
    const uint32_t off = col ? 0u : hoff[i], cap = col ? 0u : hoff[i + 1] - off;
    if (!col)
        for (uint32_t q = lane; q < cap; q += 32) hkv[off + q] = make_int2(-1, 0);
    __syncwarp();
    for (int j8 = 0; j8 < B; j8 += 32 * 8) {
        uint32_t x8[8];  // eight chunks of the row (or column) in flight
#pragma unroll
        for (int cq = 0; cq < 8; ++cq) {
            const int j = j8 + 32 * cq + lane;
            x8[cq] = j < B ? (uint32_t)(col ? cells[j * B + i] : cells[i * B + j]) : 0u;
        }
#pragma unroll
        for (int cq = 0; cq < 8; ++cq) {
            const int j0 = j8 + 32 * cq;
            if (j0 >= B) break;
            const int j = j0 + lane;
            const uint32_t v = x8[cq];
            const unsigned nz = __ballot_sync(0xffffffffu, v != 0);
            uint32_t incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (v != 0) {
                const uint32_t q = p + (uint32_t)__popc(nz & ((1u << lane) - 1u));
                if (col) {
                    cr[q] = j;
                    cv[q] = (int32_t)v;
                    cpre[q] = carry + incl;
                } else {
                    rc[q] = j;
                    rv[q] = (int32_t)v;
                    rpre[q] = carry + incl;
                    if ((int64_t)v < XT) f += T[v];
                    else fb += (double)v * log((double)v);
                    uint32_t h = sparse_hash(j) & (cap - 1);
                    bool done = false;
                    for (uint32_t t = 0; t < cap; ++t) {
                        if (atomicCAS(&hkv[off + h].x, -1, j) == -1) {
                            hkv[off + h].y = (int32_t)v;
                            done = true;
                            break;
                        }
                        h = (h + 1) & (cap - 1);
                    }
                    if (!done) record_status(status, SBP_EHASHFULL);
                }
            }
            p += (uint32_t)__popc(nz);
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    f = warp_sum_128(f);
    fb = warp_sum(fb);
    if (lane == 0) {
        (col ? din : dout)[i] = (int32_t)carry;
        if ((int64_t)carry < XT) f -= T[carry];
        else fb -= (double)carry * log((double)carry);
        lpart[w] = f;
        lfb[w] = fb;
    }
}

// (4) one CTA: per-block scalars and DL from the warps' shares of L (fixed
// order, exact)
__global__ void __launch_bounds__(kSmallThreads) k_small_finish(const int32_t *__restrict__ dout,
                                                                const int32_t *__restrict__ din, int B,
                                                                const __int128 *__restrict__ lpart,
                                                                const double *__restrict__ lfb,
                                                                int32_t *__restrict__ dsum, double *__restrict__ rcp,
                                                                float *__restrict__ rcp32, int64_t E, int64_t N,
                                                                double *__restrict__ dl) {
    __shared__ __int128 red[kSmallThreads / 32];
    __shared__ double redd[kSmallThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    __int128 f = 0;
    double fb = 0.0;
    for (int u = tid; u < B; u += kSmallThreads) {
        const int64_t d = (int64_t)dout[u] + din[u];
        dsum[u] = (int32_t)d;
        rcp[u] = 1.0 / ((double)d + (double)B);
        rcp32[u] = 1.0f / ((float)d + (float)B);
    }
    for (int q = tid; q < 2 * B; q += kSmallThreads) {
        f += lpart[q];
        fb += lfb[q];
    }
    f = warp_sum_128(f);
    fb = warp_sum(fb);
    if (lane == 0) {
        red[w] = f;
        redd[w] = fb;
    }
    __syncthreads();
    if (tid == 0) {
        __int128 L = 0;
        double Lb = 0.0;
        for (int q = 0; q < kSmallThreads / 32; ++q) {
            L += red[q];
            Lb += redd[q];
        }
        dl[0] = dl_eq2(E, N, B, fix_to_double(L) + Lb);
    }
}

template <class T>
int alloc(sbp_model *m, T **p, int64_t count) {
    model_free(*p, m->stream);
    *p = nullptr;
    if (model_alloc((void **)p, (size_t)(count > 0 ? count : 1) * sizeof(T), m->stream) != cudaSuccess) {
        cudaGetLastError();
        return fail(SBP_ENOMEM, "cudaMalloc failed for the sparse blockmodel");
    }
    return SBP_OK;
}

// the 32 pivots of every row (threads [0, 32 B)) and column (threads
// [32 B, 64 B)) of the sparse M: pivot i is the row's inclusive prefix at the
// end of its i-th segment of ceil(len / 32) entries, all ones past the row
__global__ void k_sparse_pivots(const uint32_t *__restrict__ rp, const uint32_t *__restrict__ rpre,
                                const uint32_t *__restrict__ cp, const uint32_t *__restrict__ cpre, int B,
                                uint32_t *__restrict__ rpc, uint32_t *__restrict__ cpc) {
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= 64 * (int64_t)B) return;
    const bool col = x >= 32 * (int64_t)B;
    const int64_t y = col ? x - 32 * (int64_t)B : x;
    const int u = (int)(y >> 5), i = (int)(y & 31);
    const uint32_t *p = col ? cp : rp;
    const uint32_t *pre = col ? cpre : rpre;
    const uint32_t lo = p[u], len = p[u + 1] - lo;
    const uint32_t step = (len + 31) / 32;
    uint32_t v = 0xffffffffu;
    if ((uint32_t)i * step < len) {
        const uint32_t end = ((uint32_t)i + 1) * step < len ? ((uint32_t)i + 1) * step : len;
        v = pre[lo + end - 1];
    }
    (col ? cpc : rpc)[y] = v;
}

}  // namespace

size_t sparse_bytes(const sbp_graph *g, int64_t B) {
    const size_t E = (size_t)std::max<int64_t>(g->m, 1), n = (size_t)g->n, b = (size_t)B;
    const size_t edges = 8 * 4 * E, tables = 8 * (4 * E + 2 * n), vertices = 8 * n;
    const size_t rows = 28 * b + 8, lists = 4 * (8 * b + 7 * (b / 1024 + 1)), pivots = 256 * b;
    const size_t small = std::min(b, (size_t)kSmallRowsB);
    return edges + tables + vertices + rows + lists + pivots + 4 * small * small + 4 * (size_t)kSparseScratch;
}

// (sparse_bytes says how much this allocates)
int ensure_sparse_capacity(sbp_model *m, int32_t B) {
    sbp_model::Sparse &S = m->sp;
    const int64_t E = m->g->m > 0 ? m->g->m : 1, n = m->g->n;
    if (S.cap_e < E) {
        SBP_TRY(alloc(m, &S.vo, n));
        SBP_TRY(alloc(m, &S.vi, n));
        SBP_TRY(alloc(m, &S.lo, E));
        SBP_TRY(alloc(m, &S.li, E));
        SBP_TRY(alloc(m, &S.rc, E));
        SBP_TRY(alloc(m, &S.rv, E));
        SBP_TRY(alloc(m, &S.rpre, E));
        SBP_TRY(alloc(m, &S.cr, E));
        SBP_TRY(alloc(m, &S.cv, E));
        SBP_TRY(alloc(m, &S.cpre, E));
        SBP_TRY(alloc(m, &S.hkv, 4 * E + 2 * n));
        SBP_TRY(alloc(m, &S.scratch, kSparseScratch));
        S.cap_e = E;
    }
    if (B <= kSmallRowsB && S.cap_cells < (int64_t)B * B) {
        SBP_TRY(alloc(m, &S.cells, (int64_t)B * B));
        S.cap_cells = (int64_t)B * B;
    }
    if (S.cap_b < B) {
        SBP_TRY(alloc(m, &S.rp, (int64_t)B + 1));
        SBP_TRY(alloc(m, &S.re, (int64_t)B));
        SBP_TRY(alloc(m, &S.cp, (int64_t)B + 1));
        SBP_TRY(alloc(m, &S.ce, (int64_t)B));
        SBP_TRY(alloc(m, &S.hoff, (int64_t)B + 1));
        SBP_TRY(alloc(m, &S.rcur, (int64_t)B));
        SBP_TRY(alloc(m, &S.ccur, (int64_t)B));
        SBP_TRY(alloc(m, &S.lists, 8 * (int64_t)B + 7 * ((int64_t)B / 1024 + 1)));
        SBP_TRY(alloc(m, &S.rpc, (int64_t)B * 32));
        SBP_TRY(alloc(m, &S.cpc, (int64_t)B * 32));
        S.cap_b = B;
    }
    return SBP_OK;
}

// Rebuild of the sparse blockmodel from m->b; fills the model's degree and
// per-block arrays.  after_pass: m->bnew holds the previous assignment, and
// cell counts kept from the previous rebuild may be updated from the moves.
// dl_done: DL is written too (else *n_parts partials of L are).
int rebuild_sparse(sbp_model *m, bool after_pass, bool *dl_done, int *n_parts) {
    const sbp_graph *g = m->g;
    sbp_model::Sparse &S = m->sp;
    const int B = m->B;
    const int64_t E = g->m;
    cudaStream_t st = m->stream;
    *dl_done = false;
    *n_parts = 0;
    if (B > kSmallRowsB) {
        S.cells_B = 0;
        return build_sparse_rows(m, n_parts);
    }
    // the B x B counts, then five kernels: lengths, offsets, rows with columns
    // and tables, scalars with DL, pivots
    if (after_pass && S.cells_B == B)
        SBP_TRY(update_cells(m, S.cells));
    else
        SBP_TRY(count_cells(m, S.cells));
    S.cells_B = B;
    uint32_t *rlen = S.scratch + 8, *clen = rlen + kSmallRowsB;
    __int128 *lpart = reinterpret_cast<__int128 *>(S.scratch + 8 + 2 * kSmallRowsB + 8);
    double *lfb = reinterpret_cast<double *>(lpart + 2 * kSmallRowsB);
    const int wgrid = (int)((2 * (int64_t)B * 32 + kT - 1) / kT);
    k_small_lengths<<<wgrid, kT, 0, st>>>(S.cells, B, rlen, clen);
    SBP_LAUNCHED();
    k_small_offsets<<<1, kSmallThreads, 0, st>>>(rlen, clen, B, S.rp, S.cp, S.hoff);
    SBP_LAUNCHED();
    k_small_fill<<<wgrid, kT, 0, st>>>(S.cells, B, S.rp, S.cp, S.hoff, S.rc, S.rv, S.rpre, S.cr, S.cv, S.cpre, S.hkv,
                                       m->dout, m->din, m->T, m->XT, lpart, lfb, m->status);
    SBP_LAUNCHED();
    k_small_finish<<<1, kSmallThreads, 0, st>>>(m->dout, m->din, B, lpart, lfb, m->dsum, m->rcp, m->rcp32, E, g->n,
                                                m->dl);
    SBP_LAUNCHED();
    k_sparse_pivots<<<(int)((64 * (int64_t)B + kT - 1) / kT), kT, 0, st>>>(S.rp, S.rpre, S.cp, S.cpre, B, S.rpc, S.cpc);
    SBP_LAUNCHED();
    S.slack = false;
    *dl_done = true;
    return SBP_OK;
}

void free_sparse(sbp_model *m) {
    sbp_model::Sparse &S = m->sp;
    void *ps[] = {S.vo, S.vi, S.lo,  S.li,      S.rc, S.rv, S.rpre, S.cr,    S.cv,    S.cpre, S.hkv, S.scratch, S.rp,
                  S.re, S.cp, S.ce,  S.hoff,    S.rcur, S.ccur, S.lists, S.cells, S.rpc, S.cpc};
    for (void *p : ps) model_free(p, m->stream);
    S = sbp_model::Sparse();
}

}  // namespace sbp
