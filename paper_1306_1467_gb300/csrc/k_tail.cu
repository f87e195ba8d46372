// The rest of a plain round after its search (Sec. 2.3 steps 2-4, and step 1 of
// the next round): shortlist, compensated re-scan, the round's stump, the weight
// update and the renormalisation, in one launch.
//
// These are a few microseconds of latency each -- a trip to memory, a reduction,
// a handful of FP64 operations -- around very little data, so k_tail is one
// cluster of 16 CTAs: what would be a kernel boundary is a cluster barrier, and
// the small results (listed features, run results, FP64 partial sums) pass
// through shared memory of the cluster.  Rounds of a graph replay, with four
// kernels (shortlist, re-scan, two updates) before and this now: 31.7 -> 27.6 us
// at 10x10 / 600, 148.5 -> 145.4 at 24x24 / 2,003, 771.5 -> 769.7 at 24x24 /
// 15,000 (where four times the SMs shared the FP64 additions before).
//
// Where its 51 k cycles go at 15,000 (clock stamps in a copy): shortlist 5.0,
// first barrier 1.4, re-scan 9.3, its combination 6.2 with a barrier, update
// part 1 9.4 (two trips to memory, then 13 dependent FP64 additions of about
// 250 cycles) and 4.9 at its barrier, sums and factors 3.5, part 2 7.2, the
// class totals 4.1.
//
// Every sum has the partition and order of the kernels in k_update.cu: 256
// samples a block, a value's threads and blocks added by one warp.
#include <cooperative_groups.h>
#include <limits.h>

#include "k_search.cuh"
#include "k_update.cuh"

namespace vjb {

namespace cg = cooperative_groups;

constexpr int kTailCtas = 16;  // above the portable 8: FP64 sums and row reads share more SMs
constexpr int kTailThreads = 512;  // and one warp that keeps the records
constexpr int kTailBlocks = (VJB_MAX_SAMPLES + kUpdateThreads - 1) / kUpdateThreads;  // update blocks
constexpr int kTailHalves = kTailThreads / kUpdateThreads;           // a CTA's threads take two at a time,
constexpr int kTailSteps = kTailBlocks / (kTailCtas * kTailHalves);  // at most four times
constexpr int kTailSlots = kTailHalves * kTailSteps;                 // blocks of a CTA
static_assert(kTailSteps * kTailHalves * kTailCtas == kTailBlocks && 2 * kTailSlots == kTailThreads / 32,
              "a warp per block of the CTA and value");
// Longest list the cluster re-scans itself.  Most rounds list one feature; a
// plateau of ties lists tens of thousands, and k_plateau takes those.
constexpr int kTailCands = 16;

struct TailShared {
    float red[kTailThreads / 32 + 1];
    Candidate best;
    RunResult runs[kTailCands * 32];
    float samples[kTailSlots][2][kUpdateThreads];
    double part_a[2][kTailBlocks], part_b[2][kTailBlocks];
    double total[2];
    double scale_hit, scale_miss;
    int32_t status;
};

// One value's partial sums over the update's blocks, added in order by one warp.
__device__ __forceinline__ double add_blocks(const double *part, int blocks, int lane) {
    double x = 0.0;
    for (int k = lane; k < blocks; k += 32) x += part[k];
    return warp_sum_d(x);
}

// Barrier of the threads that hold samples (all but the keeper's warp).
__device__ __forceinline__ void sample_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kTailThreads) : "memory"); }

// The CTA's blocks' sums of two values: warp 2 s + v adds value v of slot s, the
// threads 32 apart first, then the lanes by a butterfly (13 dependent FP64
// additions, side by side for all the blocks).  Every lane gets its warp's sum.
__device__ __forceinline__ double block_sum(const TailShared &S, int warp, int lane) {
    const float *x = S.samples[warp >> 1][warp & 1];
    double sum = 0.0;
#pragma unroll
    for (int q = 0; q < kUpdateThreads / 32; ++q) sum += (double)x[lane + 32 * q];
    return warp_sum_d(sum);
}

__global__ void __launch_bounds__(kTailThreads + 32, 1)
    k_tail(const __grid_constant__ JobDesc J, const float *__restrict__ bmin, int nbmin) {
    __shared__ TailShared S;
    auto cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    TailShared *lead = cluster.map_shared_rank(&S, 0);
    RoundState *rs = J.rs;

    // ---- shortlist: everything it reads is asked for at once
    constexpr int kPre = 6;
    const bool keeper = warp == kTailThreads / 32;
    const int64_t stride = kTailCtas * kTailThreads, quads = keeper ? 0 : J.nfeat >> 2, first = rank * kTailThreads + tid;
    const float4 *err4 = reinterpret_cast<const float4 *>(J.ferr);
    float4 pre[kPre];
#pragma unroll
    for (int q = 0; q < kPre; ++q)
        if (first + q * stride < quads) pre[q] = err4[first + q * stride];
    float m = INFINITY;
    for (int i = tid; i < nbmin; i += (int)blockDim.x) m = fminf(m, bmin[i]);
    const int32_t status = rs->status, forced = rs->forced, r0 = rs->rounds;
    if (status != VJB_OK || forced) return;  // the whole cluster
    m = warp_min(m);
    if (lane == 0) S.red[warp] = m;
    __syncthreads();
    m = INFINITY;
#pragma unroll
    for (int w = 0; w < kTailThreads / 32 + 1; ++w) m = fminf(m, S.red[w]);
    const float thr = shortlist_threshold(m, rs);
    auto test = [&](float e, int64_t f) {
        if (e <= thr) J.cand_ids[atomicAdd(&rs->cand_count, 1)] = (int32_t)f;  // (the count is zero between rounds)
    };
    auto test4 = [&](const float4 &e, int64_t q) {
        if (fminf(fminf(e.x, e.y), fminf(e.z, e.w)) <= thr) {
            test(e.x, 4 * q);
            test(e.y, 4 * q + 1);
            test(e.z, 4 * q + 2);
            test(e.w, 4 * q + 3);
        }
    };
#pragma unroll
    for (int q = 0; q < kPre; ++q)
        if (first + q * stride < quads) test4(pre[q], first + q * stride);
    for (int64_t q = first + kPre * stride; q < quads; q += stride) test4(err4[q], q);
    if (rank == 0 && tid < (int)(J.nfeat & 3)) test(J.ferr[(J.nfeat & ~(int64_t)3) + tid], (J.nfeat & ~(int64_t)3) + tid);
    cluster.sync();
    const int count = __ldcg(&rs->cand_count);
    if (count == 0 || count > kTailCands) {  // a long list is k_plateau's
        if (rank == 0 && tid == 0) {
            rs->screen_min = m;
            if (count == 0) {  // nothing was listed: stop the job with an error flag
                rs->flags |= kFlagNoCandidate;
                rs->status = VJB_EDEVICE;
            }
        }
        return;  // the whole cluster
    }

    // ---- compensated re-scan: a warp per run, a feature's 32 runs on 16 SMs
    for (int i = rank + kTailCtas * warp; !keeper && i < count * 32; i += kTailCtas * (kTailThreads / 32)) {
        const int32_t f = __ldcg(J.cand_ids + (i >> 5));
        const RunResult r = rescan_run(J.rows + (size_t)f * J.npad, J.npad / 32, i & 31, J.v, lane);
        if (lane < kTailCtas) cluster.map_shared_rank(&S, lane)->runs[i] = r;  // to every CTA
    }
    cluster.sync();
    // the stump, found by every CTA for itself
    if (warp == 0) {
        Candidate b;
        b.err_hi = INFINITY; b.err_lo = 0.f; b.feature = INT_MAX; b.split = INT_MAX; b.polarity = 1; b.pad = 0;
        for (int c = 0; c < count; ++c) {
            const Candidate cd = combine_runs(J, __ldcg(J.cand_ids + c), S.runs[c * 32 + lane], lane);
            if (lane == 0 && cand_less(cd, b)) b = cd;
        }
        if (lane == 0) S.best = b;
    }
    __syncthreads();
    const Candidate best = S.best;
    if (best.feature == INT_MAX) {
        if (rank == 0 && tid == 0) {
            rs->screen_min = m;
            rs->flags |= kFlagNoCandidate;
            rs->status = VJB_EDEVICE;
        }
        cluster.sync();
        return;
    }

    // ---- update, part 1: e_i of the samples in value order, FP64 sums of the
    // misclassified and of all weight.  Block b is step b / 32's, CTA (b / 2) mod
    // 16's, half b mod 2's.
    const int n = J.lay.n, blocks = (n + kUpdateThreads - 1) / kUpdateThreads;
    const int half = tid / kUpdateThreads, t = tid % kUpdateThreads;
    const int slot_blk = (warp >> 2) * (kTailCtas * kTailHalves) + rank * kTailHalves + ((warp >> 1) & 1);
    auto block_of = [&](int step) { return step * (kTailCtas * kTailHalves) + rank * kTailHalves + half; };
    int32_t theta = 0;
    if (keeper && rank == kTailCtas - 1 && lane == 0)
        theta = stump_threshold(J, best.feature, best.polarity, best.split);
#pragma unroll
    for (int step = 0; step < kTailSteps && !keeper; ++step) {
        const int k = block_of(step) * kUpdateThreads + t;
        float mw = 0.f, tw = 0.f;
        if (k < n) {
            const int i = sample_at(J, best.feature, k);
            const bool below = k < best.split, h = best.polarity > 0 ? below : !below;
            const bool miss = h != (J.y[i] != 0);
            J.miss[i] = miss;
            tw = J.w[i];
            if (miss) mw = tw;
        }
        S.samples[step * kTailHalves + half][0][t] = mw;
        S.samples[step * kTailHalves + half][1][t] = tw;
    }
    if (!keeper) sample_barrier();
    if (!keeper && slot_blk < blocks) {
        const double x = block_sum(S, warp, lane);
        if (lane < kTailCtas) cluster.map_shared_rank(&S, lane)->part_a[warp & 1][slot_blk] = x;
    }
    // part 2's weights and labels, on their way while the sums meet
    float w0[kTailSteps];
    bool face[kTailSteps];
#pragma unroll
    for (int step = 0; step < kTailSteps; ++step) {
        const int i = block_of(step) * kUpdateThreads + t;
        const bool in = !keeper && i < n;
        w0[step] = in ? J.w[i] : 0.f;
        face[step] = in && J.y[i] != 0;
    }
    cluster.sync();
    if (warp < 2) {
        const double x = add_blocks(S.part_a[warp], blocks, lane);
        if (lane == 0) S.total[warp] = x;
    }
    bool miss[kTailSteps];
#pragma unroll
    for (int step = 0; step < kTailSteps; ++step) {
        const int i = block_of(step) * kUpdateThreads + t;
        miss[step] = !keeper && i < n && __ldcg(J.miss + i) != 0;  // (written by other CTAs)
    }
    __syncthreads();
    const double M = S.total[0], T = S.total[1];
    if (tid < 2) {
        // the error, and the two factors of reweighting and renormalisation,
        // one to a thread: beta / Z for a hit, 1 / Z for a miss
        const double eps = M / T, beta = eps / (1.0 - eps), Z = M + beta * (T - M);
        const double scale = (tid ? 1.0 : beta) / Z;
        if (tid == 0) {
            S.scale_hit = scale;
            S.status = eps == 0.0 ? VJB_DONE_PERFECT : (eps >= 0.5 ? VJB_DONE_NOGAIN : VJB_OK);
        } else {
            S.scale_miss = scale;
        }
    }
    __syncthreads();
    const int32_t outcome = S.status;
    if (keeper) {
        // the records, off the path of the weights: the keeper of the last CTA
        // arrives at the barrier below, writes them, and then waits there
        if (outcome == VJB_OK) cluster.barrier_arrive();
        if (rank == kTailCtas - 1) {
            const double eps = M / T;
            if (lane == 0) {
                const vjb_stump st = stump_record(best.feature, best.polarity, theta, best.split, eps);
                *J.last = st;
                if (eps < 0.5 && r0 < J.stump_cap) J.stumps[r0] = st;
            } else if (lane == 1) {
                // what the search saw of this stump, next to its FP64 error; the
                // search works in units of the weight total T, so divide by it
                vjb_round_diag dg;
                dg.search_error = ((double)best.err_hi + (double)best.err_lo) / T;
                dg.screen_error = (float)((double)J.ferr[best.feature] / T);
                dg.screen_min = (float)((double)m / T);
                dg.candidates = count;
                dg.forced = 0;
                if (r0 < J.stump_cap) J.diag[r0] = dg;
            } else if (lane == 2) {
                rs->screen_min = m;
                rs->last_cands = count;
                rs->cand_count = 0;
                if (outcome != VJB_DONE_NOGAIN) rs->rounds = r0 + 1;
                rs->status = outcome;
            }
        }
        if (outcome == VJB_OK) cluster.barrier_wait();
        return;
    }
    if (outcome != VJB_OK) return;  // the whole cluster; its shared memory is not read from outside any more

    // ---- update, part 2: the weights and their class totals
    const double scale_hit = S.scale_hit, scale_miss = S.scale_miss;
#pragma unroll
    for (int step = 0; step < kTailSteps; ++step) {
        const int i = block_of(step) * kUpdateThreads + t;
        float fw = 0.f;
        if (i < n) {
            fw = __double2float_rn((double)w0[step] * (miss[step] ? scale_miss : scale_hit));
            J.w[i] = fw;
            store_v(J.v, J.lay, i, face[step] ? fw : -fw);
        }
        S.samples[step * kTailHalves + half][0][t] = face[step] ? fw : 0.f;
        S.samples[step * kTailHalves + half][1][t] = face[step] ? 0.f : fw;
    }
    sample_barrier();
    if (slot_blk < blocks) {
        const double x = block_sum(S, warp, lane);
        if (lane == 0) lead->part_b[warp & 1][slot_blk] = x;
    }
    cluster.sync();
    if (rank != 0) return;
    if (warp < 2) {
        const double x = add_blocks(S.part_b[warp], blocks, lane);
        if (lane == 0) S.total[warp] = x;
    }
    sample_barrier();
    if (tid == 0) {
        rs->t_pos = S.total[0];
        rs->t_neg = S.total[1];
        rs->weight_sum = S.total[0] + S.total[1];
    }
}

// A list too long for the cluster (a plateau of ties: every feature whose best
// split is the empty one has the same error): one CTA re-scans a feature at a
// time, over the whole GPU, and the CTA that finishes the last one picks the
// stump and updates the weights by itself.  In other rounds every CTA leaves
// after one read.  A round with all 78,460 features of 20x20 / 19,997 on its
// list: 6.0 ms (16.8 with a quarter of the CTAs, 44.5 by the 32 that served all
// rounds at first).
__global__ void __launch_bounds__(kUpdateThreads) k_plateau(const __grid_constant__ JobDesc J) {
    RoundState *rs = J.rs;
    const int32_t status = rs->status, count = rs->cand_count;
    if (status != VJB_OK || count == 0) return;
    __shared__ RunResult runs[32];
    __shared__ bool last;
    for (int c = blockIdx.x; c < count; c += (int)gridDim.x) {
        const Candidate cd = rescan_feature(J, J.cand_ids[c], runs);
        if (threadIdx.x == 0) {
            J.cands[c] = cd;
            __threadfence();
            last = atomicAdd(&rs->done_rescan, 1u) == (uint32_t)count - 1;
        }
        __syncthreads();
        if (last) {
            __threadfence();
            select_stump(J, count);
            const int blocks = (J.lay.n + kUpdateThreads - 1) / kUpdateThreads;
            for (int blk = 0; blk < blocks; ++blk) {
                if (!update_a_block(J, blk, false)) return;  // no stump
                __syncthreads();
            }
            if (threadIdx.x == 0) store_threshold(J);
            __syncthreads();
            finish_a(J, blocks);
            __syncthreads();
            for (int blk = 0; blk < blocks; ++blk) {
                if (!update_b_block(J, blk, false)) return;  // training is over
                __syncthreads();
            }
            finish_b(J, blocks);
            return;
        }
        __syncthreads();
    }
}

cudaError_t set_tail_limits() {
    return cudaFuncSetAttribute(k_tail, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

cudaError_t launch_tail(const JobDesc &J, const float *bmin, int nbmin, int sms, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kTailCtas);
    cfg.blockDim = dim3(kTailThreads + 32);
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kTailCtas;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_tail, J, bmin, nbmin);
    if (e != cudaSuccess) return e;
    k_plateau<<<sms * 4, kUpdateThreads, 0, st>>>(J);
    return cudaGetLastError();
}

}  // namespace vjb
