// merge.cu -- block-merge proposals and merge Delta DL (Alg. 1, Alg. 4): a
// team of warps per block; the proposal, the Delta DL terms and the choice
// of the best proposal are in merge_dev.cuh.  Then their application, and
// the compaction's map, by one cluster (merge_apply.cuh).
#include "merge_apply.cuh"

namespace sbp {
namespace {

constexpr int kMergeThreads = 256;
constexpr int kMergeWarps = kMergeThreads / 32;
// sparse blocks with more entries than this get a CTA (a hub's block of the
// first phases has thousands, and one warp on it would be the launch's tail).
// The line, in us, at 128, 512, 2048 and never: 200,000 vertices, 4M edges, heavy
// tail, one block per vertex 1760 / 1740 / 1733 / 2834, 50,000 blocks 2840 /
// 1693 / 1881 / 2435; 50,000 vertices, 6000 blocks 537 / 414 / 539 / 614; 1M
// vertices, 10M edges, 250,000 blocks 5405 / 4201 / 4371 / 6411.  Where all
// blocks have much the same entries a warp each is better (200,000 vertices,
// 6000 blocks 1576 / 1579 / 1393 / 1312).
constexpr uint32_t kMergeLong = 512;

// Teams of `parts` warps (1, 2, 4 or 8) take the blocks in turn.  long_pass
// 0: the blocks 0 .. B-1; with `longs`, blocks of more than kMergeLong
// entries are only listed there.  long_pass 1: the listed blocks.
template <bool SPARSE>
__global__ void __launch_bounds__(kMergeThreads) k_merge_proposals(ModelDev md, uint64_t seed, uint64_t round_id, int x,
                                                                   int parts, int32_t *__restrict__ longs,
                                                                   unsigned *__restrict__ n_long, int long_pass,
                                                                   int32_t *__restrict__ best_s,
                                                                   double *__restrict__ best_d) {
    __shared__ int2 queue[kMergeWarps][kMergeQueue];
    __shared__ __int128 s_fix[kMergeWarps][32];
    __shared__ double s_fb[kMergeWarps][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int team = wid / parts, part = wid - team * parts, teams = kMergeWarps / parts;
    const int64_t count = long_pass ? (int64_t)*(volatile unsigned *)n_long : md.B;
    for (int64_t base = (int64_t)blockIdx.x * teams; base < count; base += (int64_t)gridDim.x * teams) {
        const int64_t at = base + team;
        bool mine = at < count;
        const int r = mine ? (long_pass ? longs[at] : (int)at) : 0;
        if (mine && !long_pass && longs) {
            const uint32_t len = md.re[r] - md.rp[r] + md.ce[r] - md.cp[r];
            if (len > kMergeLong) {
                if (lane == 0) longs[atomicAdd(n_long, 1u)] = r;  // parts == 1 here
                mine = false;
            }
        }
        if (parts == 1 && !mine) continue;  // no barrier in a one-warp team
        // (teams of several warps meet at the barriers below; one without a
        // block works on block 0 and drops the result)
        int bs;
        double bd;
        merge_best<SPARSE>(md, seed, round_id, x, r, part, parts, queue[wid], [&](MergeSum &sum) {
            if (parts == 1) return;
            s_fix[wid][lane] = sum.fix;
            s_fb[wid][lane] = sum.fb;
            __syncthreads();
            if (part == 0)
                for (int w = 1; w < parts; ++w) {
                    sum.fix += s_fix[wid + w][lane];
                    sum.fb += s_fb[wid + w][lane];
                }
            __syncthreads();
        }, bs, bd);
        if (mine && part == 0 && lane == 0) {
            best_s[r] = bs;
            best_d[r] = bd;
        }
    }
}

// The application of a merge round: one launch of one block or one cluster;
// res (host memory): [0] the links made, [1] the new block count.
// The line between the two lies where they meet: one merge phase of B blocks
// (B / 3 merges, 4 B edges) took, with the block and with the cluster, 165
// and 221 us at 1024, 345 and 384 us at 4096, 420 and 407 us at 8192, 708 and
// 530 us at 20,000, 6.67 and 2.09 ms at 200,000.
constexpr int kApplyThreads = 1024;
constexpr int kOneCtaB = 4096;
constexpr int kApplyCluster = 8;

template <bool CLUSTER>
__global__ void __launch_bounds__(kApplyThreads) k_merge_apply(MergeApply w, uint32_t *words, int B,
                                                               const int32_t *__restrict__ best_s,
                                                               const double *__restrict__ best_d, int want,
                                                               int32_t *map, int32_t *res) {
    __shared__ TeamShared sh;
    int done, B_new;
    if constexpr (CLUSTER) {
        ClusterTeam t{sh, words};
        done = merge_apply(t, w, B, best_s, best_d, want, map, B_new);
    } else {
        CtaTeam t{sh};
        done = merge_apply(t, w, B, best_s, best_d, want, map, B_new);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        res[0] = done;
        res[1] = B_new;
    }
}

template <bool CLUSTER>
__global__ void __launch_bounds__(kApplyThreads) k_compact_map(uint32_t *words, int B,
                                                               const int32_t *__restrict__ present, int32_t *map,
                                                               int32_t *res) {
    __shared__ TeamShared sh;
    int B_new;
    if constexpr (CLUSTER) {
        ClusterTeam t{sh, words};
        B_new = compact_map(t, B, present, map);
    } else {
        CtaTeam t{sh};
        B_new = compact_map(t, B, present, map);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) res[1] = B_new;
}

// the work arrays of both kernels, for B blocks
int ensure_merge_work(sbp_model *m, int32_t B) {
    if (m->merge_work_B >= B) return SBP_OK;
    model_free(m->merge_work, m->stream);
    m->merge_work = nullptr;
    m->merge_work_B = 0;
    if (model_alloc((void **)&m->merge_work, merge_work_bytes(B), m->stream) != cudaSuccess) {
        cudaGetLastError();
        return fail(SBP_ENOMEM, "device allocation failed for the merge phase");
    }
    m->merge_work_B = B;
    return SBP_OK;
}

struct MergeWork {
    MergeApply w;
    uint32_t *words;
};

MergeWork merge_work(const sbp_model *m) {
    const size_t B = (size_t)m->merge_work_B;
    MergeWork x;
    x.w.key = reinterpret_cast<unsigned long long *>(m->merge_work);
    int32_t *p = reinterpret_cast<int32_t *>(x.w.key + B);
    x.w.a0 = p;
    x.w.a1 = p + B;
    x.w.x0 = p + 2 * B;
    x.w.x1 = p + 3 * B;
    x.w.mark = p + 4 * B;
    x.words = reinterpret_cast<uint32_t *>(p + 5 * B);
    return x;
}

}  // namespace

size_t merge_work_bytes(int64_t B) { return (size_t)B * kMergeApplyBytes + kClusterWords * 4; }

int launch_merge_proposals(sbp_model *m, uint64_t round_id) {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int x = m->p.merge_proposals;
    const ModelDev md = model_dev(m);
    // warps per block: enough teams to fill the chip (B blocks on sms * 32
    // warps); a dense row of a few hundred blocks also shortens with more
    int parts = 1;
    while (parts < kMergeWarps && (int64_t)m->B * parts < (int64_t)sms * 32) parts *= 2;
    int32_t *longs = nullptr;
    unsigned *n_long = reinterpret_cast<unsigned *>(m->status + 3);
    if (md.sparse && parts == 1) {
        longs = m->vcount;  // scratch of the compaction, free during a merge
        SBP_CUDA(cudaMemsetAsync(n_long, 0, 4, m->stream));
    }
    const int teams = kMergeWarps / parts;
    const int64_t blocks = ((int64_t)m->B + teams - 1) / teams;
    const int grid = (int)(blocks < (int64_t)sms * 8 ? blocks : (int64_t)sms * 8);
    const auto kern = md.sparse ? k_merge_proposals<true> : k_merge_proposals<false>;
    kern<<<grid, kMergeThreads, 0, m->stream>>>(md, m->p.seed, round_id, x, parts, longs, n_long, 0,
                                                             m->best_s, m->best_d);
    SBP_LAUNCHED();
    if (longs) {
        kern<<<sms * 4, kMergeThreads, 0, m->stream>>>(md, m->p.seed, round_id, x, kMergeWarps, longs,
                                                                    n_long, 1, m->best_s, m->best_d);
        SBP_LAUNCHED();
    }
    return SBP_OK;
}

// The round's best proposals applied on the device: m->map and, on the host,
// the links made (at most want) and the new block count.
int apply_merge_round(sbp_model *m, int32_t want, int32_t *done, int32_t *B_new) {
    SBP_TRY(ensure_merge_work(m, m->B));
    const MergeWork x = merge_work(m);
    const bool cl = m->B > kOneCtaB;
    int32_t *h = static_cast<int32_t *>(m->pinned);  // (written by the kernel)
    SBP_TRY(launch_cluster(cl ? k_merge_apply<true> : k_merge_apply<false>, cl ? kApplyCluster : 1, kApplyThreads, 0,
                           m->stream, 1, x.w, x.words, (int)m->B, (const int32_t *)m->best_s,
                           (const double *)m->best_d, (int)want, m->map, h));
    SBP_CUDA(cudaStreamSynchronize(m->stream));
    *done = h[0];
    *B_new = h[1];
    return SBP_OK;
}

// m->map for dropping the blocks without vertices; *B_new their number left
int compact_blocks(sbp_model *m, int32_t *B_new) {
    SBP_TRY(launch_vertex_count(m));
    const bool cl = m->B > kOneCtaB;
    if (cl) SBP_TRY(ensure_merge_work(m, m->B));
    uint32_t *words = cl ? merge_work(m).words : nullptr;  // (a block alone exchanges nothing)
    int32_t *h = static_cast<int32_t *>(m->pinned);        // (written by the kernel)
    SBP_TRY(launch_cluster(cl ? k_compact_map<true> : k_compact_map<false>, cl ? kApplyCluster : 1, kApplyThreads, 0,
                           m->stream, 1, words, (int)m->B, (const int32_t *)m->vcount, m->map, h));
    SBP_CUDA(cudaStreamSynchronize(m->stream));
    *B_new = h[1];
    return SBP_OK;
}

}  // namespace sbp
