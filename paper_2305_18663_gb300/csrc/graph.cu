// graph.cu -- graph upload: directed COO -> CSR of out-edges and of in-edges.
//
// The graph is the fixed input "Graph G" of Alg. 1-2.  Rows are sorted by
// neighbour id (the order the nodal proposal indexes into), duplicates and
// self-loops are kept.  Vertices are also grouped by total degree so the
// nodal pass can give small, medium and large rows different work units;
// the grouping changes no result (every decision reads frozen state only).
//
// The whole build runs on the device: the out-rows come from a radix sort of
// the (source, target) keys, the in-rows from a stable sort of the out-rows'
// positions by target, the two vertex orders from stable sorts on the degree.
// It is bound by the copies from pageable host memory and the sorts' passes:
// 5M edges of 300k vertices take 1.47 ms from the host, 1.24 ms from the device
// (counted and sorted on the host cores, 113 ms).
#include <algorithm>
#include <string>

#include "common.cuh"

namespace sbp {
namespace {

constexpr int kT = 256;

// memory the build's kernels read where it lies: of the current device, or
// managed (anything else is copied)
bool readable_in_place(const void *p) {
    cudaPointerAttributes a;
    int dev = 0;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (a.type == cudaMemoryTypeDevice && a.device == dev) || a.type == cudaMemoryTypeManaged;
}

int grid_of(int64_t work) {
    const int64_t g = (work + kT - 1) / kT;
    return (int)(g < 1 ? 1 : g > 152 * 16 ? 152 * 16 : g);
}

int bits_for(uint64_t maxval) {
    int b = 1;
    while (b < 64 && (maxval >> b) != 0) ++b;
    return b;
}

// what the host needs to know of the graph
struct Info {
    unsigned long long bad;  // the first edge with an id out of range (all ones: none)
    unsigned long long cnt[6];  // vertices of the degree groups, the top one in its three classes
    unsigned long long n_self;
    int32_t maxk;
};

// the edge (s, d) as one key, and the first edge with an id outside [0, n)
// (its key is made from vertex 0, so that what follows stays in range)
template <class K>
__global__ void __launch_bounds__(kT) k_edge_keys(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                                                  int64_t m, int64_t n, K *__restrict__ keys, Info *__restrict__ info) {
    for (int64_t e = (int64_t)blockIdx.x * kT + threadIdx.x; e < m; e += (int64_t)gridDim.x * kT) {
        int64_t s = src[e], d = dst[e];
        if (s < 0 || s >= n || d < 0 || d >= n) {
            atomicMin(&info->bad, (unsigned long long)e);
            s = d = 0;
        }
        keys[e] = (K)((uint64_t)s * (uint64_t)n + (uint64_t)d);
    }
}

// sorted keys -> out-rows, and the sort key (target) and value (position)
// of the in-rows
template <class K>
__global__ void __launch_bounds__(kT) k_out_rows(const K *__restrict__ keys, int64_t m, int64_t n,
                                                 int32_t *__restrict__ oc, int32_t *__restrict__ esrc,
                                                 uint32_t *__restrict__ ikey, uint32_t *__restrict__ ival) {
    for (int64_t e = (int64_t)blockIdx.x * kT + threadIdx.x; e < m; e += (int64_t)gridDim.x * kT) {
        const uint64_t k = (uint64_t)keys[e], s = k / (uint64_t)n;
        const uint32_t d = (uint32_t)(k - s * (uint64_t)n);
        esrc[e] = (int32_t)s;
        oc[e] = (int32_t)d;
        ikey[e] = d;
        ival[e] = (uint32_t)e;
    }
}

// in-row position j holds out-edge e = ival[j] (its keys and values are idst
// and tw_io).  The sort is stable and the out-rows are ascending, so in-rows
// are ascending too and the k-th copy of a repeated edge is paired with its
// k-th copy.
__global__ void __launch_bounds__(kT) k_in_rows(const uint32_t *__restrict__ ikey, const uint32_t *__restrict__ ival,
                                                const int32_t *__restrict__ esrc, int64_t m, int32_t *__restrict__ ic,
                                                int32_t *__restrict__ tw_oi, Info *__restrict__ info) {
    for (int64_t j = (int64_t)blockIdx.x * kT + threadIdx.x; j < m; j += (int64_t)gridDim.x * kT) {
        const uint32_t e = ival[j];
        const int32_t s = esrc[e];
        ic[j] = s;
        tw_oi[e] = (int32_t)j;
        if ((uint32_t)s == ikey[j]) atomicAdd(&info->n_self, 1ull);
    }
}

__global__ void __launch_bounds__(kT) k_self_loops(const uint32_t *__restrict__ ikey, const int32_t *__restrict__ ic,
                                                   int64_t m, unsigned *__restrict__ count,
                                                   int32_t *__restrict__ self_in) {
    for (int64_t j = (int64_t)blockIdx.x * kT + threadIdx.x; j < m; j += (int64_t)gridDim.x * kT)
        if ((uint32_t)ic[j] == ikey[j]) self_in[atomicAdd(count, 1u)] = (int32_t)j;
}

// row offsets by binary search in the sorted row ids (both CSRs): ptr[v] is
// the first position whose row is not below v
template <class R>
__device__ __forceinline__ int32_t first_not_below(const R *__restrict__ row, int64_t m, int64_t v) {
    int64_t lo = 0, len = m;
    while (len > 0) {
        const int64_t half = len >> 1;
        if ((int64_t)row[lo + half] < v) {
            lo += half + 1;
            len -= half + 1;
        } else {
            len = half;
        }
    }
    return (int32_t)lo;
}

__global__ void __launch_bounds__(kT) k_row_offsets(const int32_t *__restrict__ esrc, const uint32_t *__restrict__ ikey,
                                                    int64_t m, int64_t n, int32_t *__restrict__ op,
                                                    int32_t *__restrict__ ip) {
    for (int64_t v = (int64_t)blockIdx.x * kT + threadIdx.x; v <= n; v += (int64_t)gridDim.x * kT) {
        op[v] = first_not_below(esrc, m, v);
        ip[v] = first_not_below(ikey, m, v);
    }
}

__device__ __forceinline__ int degree_group(int32_t k) {
    return k == 0 ? 0 : k <= kSmallDeg ? 1 : k <= kWarpDeg ? 2 : 3;
}

__device__ __forceinline__ int degree_class(int32_t k) {
    return k <= kWarpDeg ? degree_group(k) : k <= kMidDeg ? 3 : k <= kWideDeg ? 4 : 5;
}

// sizes of the degree classes and the largest degree
__global__ void __launch_bounds__(kT) k_degree_classes(const int32_t *__restrict__ op, const int32_t *__restrict__ ip,
                                                       int64_t n, Info *__restrict__ info) {
    __shared__ unsigned cnt[6];
    __shared__ int mx;
    if (threadIdx.x < 6) cnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) mx = 0;
    __syncthreads();
    int m = 0;
    unsigned c[6] = {0, 0, 0, 0, 0, 0};
    for (int64_t v = (int64_t)blockIdx.x * kT + threadIdx.x; v < n; v += (int64_t)gridDim.x * kT) {
        const int32_t k = (op[v + 1] - op[v]) + (ip[v + 1] - ip[v]);
        m = max(m, k);
        const int q = degree_class(k);
#pragma unroll
        for (int i = 0; i < 6; ++i) c[i] += q == i;
    }
    m = __reduce_max_sync(0xffffffffu, m);
#pragma unroll
    for (int i = 0; i < 6; ++i) c[i] = __reduce_add_sync(0xffffffffu, c[i]);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&mx, m);
        for (int i = 0; i < 6; ++i) atomicAdd(&cnt[i], c[i]);
    }
    __syncthreads();
    if (threadIdx.x < 6 && cnt[threadIdx.x]) atomicAdd(&info->cnt[threadIdx.x], (unsigned long long)cnt[threadIdx.x]);
    if (threadIdx.x == 0) atomicMax(&info->maxk, mx);
}

// sort keys of a vertex order (both stable, so ties keep id order): by group
// with the top group by descending degree, or all by descending degree
__global__ void __launch_bounds__(kT) k_order_keys(const int32_t *__restrict__ op, const int32_t *__restrict__ ip,
                                                   int64_t n, int32_t maxk, bool groups, uint32_t *__restrict__ key,
                                                   uint32_t *__restrict__ val) {
    for (int64_t v = (int64_t)blockIdx.x * kT + threadIdx.x; v < n; v += (int64_t)gridDim.x * kT) {
        const int32_t k = (op[v + 1] - op[v]) + (ip[v + 1] - ip[v]);
        const int q = groups ? degree_group(k) : 3;
        key[v] = q < 3 ? (uint32_t)q : 3u + (uint32_t)(maxk - k);
        val[v] = (uint32_t)v;
    }
}

// carves aligned arrays out of one allocation
struct Carver {
    unsigned char *p = nullptr;
    size_t used = 0;
    template <class T>
    void take(T **out, size_t count) {
        if (p) *out = reinterpret_cast<T *>(p + used);
        used += ((count > 0 ? count : 1) * sizeof(T) + 255) / 256 * 256;
    }
};

// The per-edge arrays are carved as three pairs, and the build sorts in them:
// nothing else of the edges' size is held while a graph is loaded.
struct Pairs {
    int32_t *p[3] = {nullptr, nullptr, nullptr};
    size_t half = 0;  // second array of a pair
};

struct Scratch {
    uint32_t *k0 = nullptr, *k1 = nullptr;  // keys and values of the vertex sorts
    uint32_t *words = nullptr;
    Info *info = nullptr;
    unsigned *count = nullptr;
};

int load_edges(int64_t m, const int32_t *from, int32_t *buf, const int32_t **use, cudaStream_t st) {
    *use = from;
    if (readable_in_place(from)) return SBP_OK;
    SBP_CUDA(cudaMemcpyAsync(buf, from, (size_t)m * 4, cudaMemcpyDefault, st));
    *use = buf;
    return SBP_OK;
}

// sorts the keys in pairs 1 and 2 and makes the out-rows; *at: the pair that
// then holds the in-rows' keys and values
template <class K>
int sort_edges(const int32_t *s, const int32_t *d, int64_t m, int64_t n, const Scratch &x, const Pairs &e, sbp_graph *g,
               int *at, cudaStream_t st) {
    K *k0 = reinterpret_cast<K *>(e.p[1]), *k1 = reinterpret_cast<K *>(e.p[2]);
    k_edge_keys<K><<<grid_of(m), kT, 0, st>>>(s, d, m, n, k0, x.info);
    SBP_LAUNCHED();
    bool first = true;
    SBP_TRY((radix_sort<K, uint32_t>(k0, k1, nullptr, nullptr, m, bits_for((uint64_t)n * (uint64_t)n - 1), x.words, st,
                                     &first)));
    // the in-rows' keys and values go where the sorted keys are not; those are
    // done with after this
    *at = first ? 2 : 1;
    uint32_t *ikey = reinterpret_cast<uint32_t *>(e.p[*at]);
    k_out_rows<K><<<grid_of(m), kT, 0, st>>>(first ? k0 : k1, m, n, g->oc, g->esrc, ikey, ikey + e.half);
    SBP_LAUNCHED();
    return SBP_OK;
}

// one vertex order
int sort_vertices(const sbp_graph *g, int32_t maxk, bool groups, const Scratch &x, int32_t *out, cudaStream_t st) {
    const size_t n = (size_t)g->n;
    uint32_t *k0 = x.k0, *k1 = x.k1;
    k_order_keys<<<grid_of(g->n), kT, 0, st>>>(g->op, g->ip, g->n, maxk, groups, k0, k0 + n);
    SBP_LAUNCHED();
    bool first = true;
    SBP_TRY((radix_sort<uint32_t, uint32_t>(k0, k1, k0 + n, k1 + n, g->n, bits_for(3u + (uint64_t)maxk), x.words, st,
                                            &first)));
    SBP_CUDA(cudaMemcpyAsync(out, (first ? k0 : k1) + n, n * 4, cudaMemcpyDeviceToDevice, st));
    return SBP_OK;
}

// everything but the self-loop positions, whose number `info` then holds
int build_graph(sbp_graph *g, const int32_t *src, const int32_t *dst, const Scratch &x, const Pairs &e, Info *info,
                uint32_t **ikey, cudaStream_t st) {
    const int64_t n = g->n, m = g->m;
    SBP_CUDA(cudaMemsetAsync(x.info, 0, sizeof(Info), st));
    SBP_CUDA(cudaMemsetAsync(&x.info->bad, 0xff, 8, st));
    *ikey = nullptr;
    // pair 0: the edge list, where it has to be copied, until its keys are
    // made; then the out-rows.  Pairs 1 and 2: the keys of the first sort and
    // its second buffer; then the in-rows' keys and values and theirs, which
    // end as idst and tw_io in one pair, with the other free for ic and tw_oi
    g->oc = e.p[0];
    g->esrc = e.p[0] + e.half;
    int at = 1;
    if (m > 0) {
        const int32_t *s, *d;
        SBP_TRY(load_edges(m, src, e.p[0], &s, st));
        SBP_TRY(load_edges(m, dst, e.p[0] + e.half, &d, st));
        if ((uint64_t)n * (uint64_t)n <= (uint64_t(1) << 32)) SBP_TRY(sort_edges<uint32_t>(s, d, m, n, x, e, g, &at, st));
        else SBP_TRY(sort_edges<uint64_t>(s, d, m, n, x, e, g, &at, st));
        uint32_t *a = reinterpret_cast<uint32_t *>(e.p[at]), *c = reinterpret_cast<uint32_t *>(e.p[3 - at]);
        bool first = true;
        SBP_TRY((radix_sort<uint32_t, uint32_t>(a, c, a + e.half, c + e.half, m, bits_for((uint64_t)n - 1), x.words, st,
                                                &first)));
        if (!first) at = 3 - at;
    }
    g->idst = e.p[at];
    g->tw_io = e.p[at] + e.half;
    g->ic = e.p[3 - at];
    g->tw_oi = e.p[3 - at] + e.half;
    if (m > 0) {
        *ikey = reinterpret_cast<uint32_t *>(g->idst);
        k_in_rows<<<grid_of(m), kT, 0, st>>>(*ikey, *ikey + e.half, g->esrc, m, g->ic, g->tw_oi, x.info);
        SBP_LAUNCHED();
    }
    k_row_offsets<<<grid_of(n + 1), kT, 0, st>>>(g->esrc, *ikey, m, n, g->op, g->ip);
    SBP_LAUNCHED();
    k_degree_classes<<<grid_of(n), kT, 0, st>>>(g->op, g->ip, n, x.info);
    SBP_LAUNCHED();
    SBP_CUDA(cudaMemcpyAsync(info, x.info, sizeof(Info), cudaMemcpyDeviceToHost, st));
    SBP_CUDA(cudaStreamSynchronize(st));
    return SBP_OK;
}

// the vertex orders and the self-loop positions, from build_graph's rows
int finish_graph(sbp_graph *g, const Scratch &x, const Info &info, const uint32_t *ikey, cudaStream_t st) {
    g->max_deg = info.maxk;
    g->bin[0] = 0;
    for (int i = 0; i < 3; ++i) g->bin[i + 1] = g->bin[i] + (int64_t)info.cnt[i];
    g->bin[4] = g->n;
    g->n_mid = (int64_t)info.cnt[3];
    g->n_wide = (int64_t)info.cnt[4];
    g->n_self = (int64_t)info.n_self;
    if (g->n_self > 0) {
        if (cudaMalloc((void **)&g->self_in, (size_t)g->n_self * 4) != cudaSuccess) {
            cudaGetLastError();
            return fail(SBP_ENOMEM, "cudaMalloc failed while loading the graph");
        }
        SBP_CUDA(cudaMemsetAsync(x.count, 0, 4, st));
        k_self_loops<<<grid_of(g->m), kT, 0, st>>>(ikey, g->ic, g->m, x.count, g->self_in);
        SBP_LAUNCHED();
    }
    SBP_TRY(sort_vertices(g, info.maxk, true, x, g->order, st));
    SBP_TRY(sort_vertices(g, info.maxk, false, x, g->by_degree, st));
    SBP_CUDA(cudaStreamSynchronize(st));
    return SBP_OK;
}

// Arrays of a graph and of its build, in one allocation each
void carve_graph(sbp_graph *g, Pairs &e, Carver &c) {
    const size_t n = (size_t)g->n;
    e.half = ((size_t)std::max<int64_t>(g->m, 1) + 63) / 64 * 64;  // (aligned as an allocation is)
    c.take(&g->op, n + 1);
    c.take(&g->ip, n + 1);
    for (auto &p : e.p) c.take(&p, 2 * e.half);
    c.take(&g->order, n);
    c.take(&g->by_degree, n);
}

void carve_scratch(Scratch &x, int64_t n, int64_t m, Carver &c) {
    c.take(&x.k0, 2 * (size_t)n);
    c.take(&x.k1, 2 * (size_t)n);
    c.take(&x.words, (size_t)sort_scratch_words(std::max(n, m)));
    c.take(&x.info, 1);
    c.take(&x.count, 1);
}

}  // namespace
}  // namespace sbp

extern "C" int sbp_load_graph(int64_t n, int64_t m, const int32_t *src, const int32_t *dst, sbp_graph_t **out) {
    using namespace sbp;
    if (!out) return fail(SBP_EINVAL, "sbp_load_graph: out is NULL");
    *out = nullptr;
    if (n < 1 || n > INT32_MAX - 1) return fail(SBP_EINVAL, "sbp_load_graph: n must be in [1, 2^31-2]");
    if (m < 0 || m >= (int64_t(1) << 30)) return fail(SBP_EINVAL, "sbp_load_graph: m must be in [0, 2^30)");
    if (m > 0 && (!src || !dst)) return fail(SBP_EINVAL, "sbp_load_graph: src/dst is NULL");
    // the legacy stream: device arrays are read behind the work that wrote them
    cudaStream_t st = nullptr;
    auto *g = new sbp_graph();
    g->n = n;
    g->m = m;
    cudaGetDevice(&g->device);
    Scratch x;
    Pairs e;
    Carver cg, cs;  // first without memory, for the sizes
    carve_graph(g, e, cg);
    carve_scratch(x, n, m, cs);
    unsigned char *scratch = nullptr;
    int rc = SBP_OK;
    if (cudaMalloc((void **)&g->slab, cg.used) != cudaSuccess ||
        model_alloc((void **)&scratch, cs.used, st) != cudaSuccess) {
        cudaGetLastError();
        rc = fail(SBP_ENOMEM, "device allocation failed while loading the graph");
    }
    if (rc == SBP_OK) {
        cg = Carver{g->slab, 0};
        cs = Carver{scratch, 0};
        carve_graph(g, e, cg);
        carve_scratch(x, n, m, cs);
        Info info{};
        uint32_t *ikey = nullptr;
        rc = build_graph(g, src, dst, x, e, &info, &ikey, st);
        if (rc == SBP_OK && info.bad != ~0ull)
            rc = fail(SBP_EINVAL, "sbp_load_graph: vertex id out of range at edge " + std::to_string(info.bad));
        if (rc == SBP_OK) rc = finish_graph(g, x, info, ikey, st);
    }
    model_free(scratch, st);
    if (rc != SBP_OK) {
        sbp_free_graph(g);
        return rc;
    }
    *out = g;
    return SBP_OK;
}

extern "C" int sbp_graph_info(const sbp_graph_t *g, int64_t *n, int64_t *m) {
    if (!g) return sbp::fail(SBP_EINVAL, "sbp_graph_info: NULL graph");
    if (n) *n = g->n;
    if (m) *m = g->m;
    return SBP_OK;
}

extern "C" void sbp_free_graph(sbp_graph_t *g) {
    if (!g) return;
    cudaFree(g->slab);
    cudaFree(g->self_in);
    delete g;
}
