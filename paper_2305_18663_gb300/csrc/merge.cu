// merge.cu -- block-merge proposals and merge Delta DL (Alg. 1, Alg. 4): a
// team of warps per block; the proposal, the Delta DL terms and the choice
// of the best proposal are in merge_dev.cuh.
#include "merge_dev.cuh"

namespace sbp {
namespace {

constexpr int kMergeThreads = 256;
constexpr int kMergeWarps = kMergeThreads / 32;
// sparse blocks with more entries than this get a CTA (a hub's block of the
// first phases has thousands, and one warp on it would be the launch's tail)
constexpr uint32_t kMergeLong = 512;

// Teams of `parts` warps (1, 2, 4 or 8) take the blocks in turn.  long_pass
// 0: the blocks 0 .. B-1; with `longs`, blocks of more than kMergeLong
// entries are only listed there.  long_pass 1: the listed blocks.
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
            const uint32_t len = md.rp[r + 1] - md.rp[r] + md.cp[r + 1] - md.cp[r];
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
        merge_best(md, seed, round_id, x, r, part, parts, queue[wid], [&](MergeSum &sum) {
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

}  // namespace

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
    k_merge_proposals<<<grid, kMergeThreads, 0, m->stream>>>(md, m->p.seed, round_id, x, parts, longs, n_long, 0,
                                                             m->best_s, m->best_d);
    SBP_LAUNCHED();
    if (longs) {
        k_merge_proposals<<<sms * 4, kMergeThreads, 0, m->stream>>>(md, m->p.seed, round_id, x, kMergeWarps, longs,
                                                                    n_long, 1, m->best_s, m->best_d);
        SBP_LAUNCHED();
    }
    return SBP_OK;
}

}  // namespace sbp
