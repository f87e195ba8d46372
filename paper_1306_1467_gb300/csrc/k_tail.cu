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
// 15,000 (where four times the SMs shared the FP64 additions before); by now, with
// less code here and a faster search, 27.2, 142.2 and 753.4.
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
constexpr int kTailHalves = kTailThreads / kUpdateThreads;  // a CTA's threads take two at a time
// Longest list the cluster re-scans itself.  Most rounds list one feature; equal
// columns list tens or hundreds and a plateau of ties tens of thousands, and
// k_plateau takes those.  After the search at 15,000 samples 15 listed features
// take 35 us here, and 21 take 43 there (windows 2 wide with equal rows).
constexpr int kTailCands = 16;
// CTAs of a k_plateau cluster: the portable 8, of which 36 clusters run at once
// (288 CTAs); of 16 only 14 fit beside each other, and a re-scan of 78,460
// features took 6.8 ms instead of 5.3.
constexpr int kPlateauCtas = 8;
static_assert(kTailCands <= kTailThreads / 32 && kTailCands >= kPlateauCtas, "a warp per listed feature, a place per CTA");

// Shared memory of a CTA in a cluster of CTAS.
template <int CTAS>
struct TailShared {
    static constexpr int kSteps = kTailBlocks / (CTAS * kTailHalves);  // at most so many times two blocks
    static constexpr int kSlots = kTailHalves * kSteps;                // blocks of a CTA
    static_assert(kSteps * kTailHalves * CTAS == kTailBlocks, "every block has one place");
    float red[kTailThreads / 32 + 1];
    Candidate found[kTailCands];  // a listed feature each (k_tail), or a CTA's best (k_plateau)
    union {
        RunResult runs[kTailCands * 32];           // until the stump is known
        float samples[kSlots][2][kUpdateThreads];  // then
    };
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

// The CTA's blocks' sums of two values: a warp adds value v of slot s, the threads
// 32 apart first, then the lanes by a butterfly (13 dependent FP64 additions, side
// by side for all the blocks).  put(v, block, sum) is called by every lane.
template <int CTAS, class Put>
__device__ __forceinline__ void block_sums(const TailShared<CTAS> &S, int rank, int blocks, int warp, int lane, Put put) {
    constexpr int kWarps = kTailThreads / 32;
#pragma unroll
    for (int k0 = 0; k0 < 2 * TailShared<CTAS>::kSlots; k0 += kWarps) {
        const int s = (k0 + warp) >> 1, v = warp & 1;
        const int blk = s / kTailHalves * (CTAS * kTailHalves) + rank * kTailHalves + s % kTailHalves;
        if (blk >= blocks) continue;
        const float *x = S.samples[s][v];
        double sum = 0.0;
#pragma unroll
        for (int q = 0; q < kUpdateThreads / 32; ++q) sum += (double)x[lane + 32 * q];
        put(v, blk, warp_sum_d(sum));
    }
}

__device__ __forceinline__ Candidate no_candidate() {
    Candidate b;
    b.err_hi = INFINITY; b.err_lo = 0.f; b.feature = INT_MAX; b.split = INT_MAX; b.polarity = 1; b.pad = 0;
    return b;
}

// The best of the first `count` places, for every thread.
__device__ __forceinline__ Candidate best_found(const Candidate *found, int count) {
    Candidate b = no_candidate();
#pragma unroll 1
    for (int k = 0; k < count; ++k)
        if (cand_less(found[k], b)) b = found[k];
    return b;
}

// The round's stump `best` of a list of `count`, chosen over a smallest screened
// error of m: its record, the weight update and the class totals, by one cluster
// whose CTAs all know the stump and no longer read the run results.  r0 rounds
// are done.
template <int CTAS>
static __device__ __forceinline__ void tail_update(const JobDesc &J, TailShared<CTAS> &S, const Candidate &best, int count,
                                                   float m, int32_t r0) {
    constexpr int kSteps = TailShared<CTAS>::kSteps;
    auto cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool keeper = warp == kTailThreads / 32;
    TailShared<CTAS> *lead = cluster.map_shared_rank(&S, 0);
    RoundState *rs = J.rs;
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
    // misclassified and of all weight.  Block b is step b / (2 CTAS)'s, CTA (b / 2)
    // mod CTAS's, half b mod 2's.
    const int n = J.lay.n, blocks = (n + kUpdateThreads - 1) / kUpdateThreads;
    const int half = tid / kUpdateThreads, t = tid % kUpdateThreads;
    auto block_of = [&](int step) { return step * (CTAS * kTailHalves) + rank * kTailHalves + half; };
    int32_t theta = 0;
    if (keeper && rank == CTAS - 1 && lane == 0)
        theta = stump_threshold(J, best.feature, best.polarity, best.split);
#pragma unroll
    for (int step = 0; step < kSteps && !keeper; ++step) {
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
    if (!keeper)
        block_sums(S, rank, blocks, warp, lane, [&](int v, int blk, double x) {
            if (lane < CTAS) cluster.map_shared_rank(&S, lane)->part_a[v][blk] = x;
        });
    // part 2's weights and labels, on their way while the sums meet
    float w0[kSteps];
    bool face[kSteps];
#pragma unroll
    for (int step = 0; step < kSteps; ++step) {
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
    bool miss[kSteps];
#pragma unroll
    for (int step = 0; step < kSteps; ++step) {
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
        if (rank == CTAS - 1) {
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
    for (int step = 0; step < kSteps; ++step) {
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
    block_sums(S, rank, blocks, warp, lane, [&](int v, int blk, double x) {
        if (lane == 0) lead->part_b[v][blk] = x;
    });
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

__global__ void __launch_bounds__(kTailThreads + 32, 1)
    k_tail(const __grid_constant__ JobDesc J, const float *__restrict__ bmin, int nbmin) {
    __shared__ TailShared<kTailCtas> S;
    auto cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    RoundState *rs = J.rs;

    // ---- shortlist: everything it reads is asked for at once, up to 24 errors a
    // thread (196,608 features; 24x24 windows have 162,336), then as many again.
    // The tail with one value after another beyond those, and now: 34 and 27 us at
    // 32x32, 65 and 35 at 48x48, 145 and 55 at 64x64 (a grid took 30, 45 and 81)
    constexpr int kPre = 6;
    const bool keeper = warp == kTailThreads / 32;
    const int stride = kTailCtas * kTailThreads, quads = keeper ? 0 : (int)(J.nfeat >> 2), first = rank * kTailThreads + tid;
    const float4 *err4 = reinterpret_cast<const float4 *>(J.ferr);
    float4 e[kPre];
    auto ask = [&](int q0) {
#pragma unroll
        for (int u = 0; u < kPre; ++u) e[u] = err4[min(q0 + u * stride, quads - 1)];
    };
    if (first < quads) ask(first);
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
    // few threads list anything: those read their four errors again, so that one
    // piece of code serves all of them (after a long search the tail's code is
    // fetched anew, and its length counts: rounds at 24x24 / 2,003 146.6 us with a
    // test for each of 14 loads and a second form of the re-scan, 142.2 now)
    for (int q0 = first; q0 < quads;) {
        uint32_t hits = 0u;
#pragma unroll
        for (int u = 0; u < kPre; ++u)
            if (q0 + u * stride < quads && fminf(fminf(e[u].x, e[u].y), fminf(e[u].z, e[u].w)) <= thr) hits |= 1u << u;
        while (hits) {
            const int q = q0 + (__ffs(hits) - 1) * stride;
            hits &= hits - 1u;
            const float4 x = err4[q];
            test(x.x, 4 * (int64_t)q);
            test(x.y, 4 * (int64_t)q + 1);
            test(x.z, 4 * (int64_t)q + 2);
            test(x.w, 4 * (int64_t)q + 3);
        }
        q0 += kPre * stride;
        if (q0 < quads) ask(q0);
    }
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

    // ---- compensated re-scan: a warp per run, a feature's 32 runs on 16 SMs (two
    // runs side by side for lists above 8 gained nothing)
    for (int i = rank + kTailCtas * warp; !keeper && i < count * 32; i += kTailCtas * (kTailThreads / 32)) {
        const int32_t f = __ldcg(J.cand_ids + (i >> 5));
        const RunResult r = rescan_run(J.rows + (size_t)f * J.npad, J.npad / 32, i & 31, J.v, lane);
        if (lane < kTailCtas) cluster.map_shared_rank(&S, lane)->runs[i] = r;  // to every CTA
    }
    cluster.sync();
    // the stump, found by every CTA for itself: a warp per feature, then a look at
    // each (15 features at 15,000 samples and at 600 take 35 and 28 us after the
    // search; 55 and 49 when one warp combined them all)
    if (warp < count) {
        const Candidate cd = combine_runs(J, __ldcg(J.cand_ids + warp), S.runs[warp * 32 + lane], lane);
        if (lane == 0) S.found[warp] = cd;
    }
    __syncthreads();
    const Candidate best = best_found(S.found, count);
    tail_update(J, S, best, count, m, r0);
}

// A list too long for one cluster (a plateau of ties: every feature whose best
// split is the empty one has the same error): every CTA of the GPU takes its share,
// up to 16 features at a time with a warp per run, and the cluster that is the
// last to finish picks the stump and updates the weights as k_tail does.  In other
// rounds every CTA leaves after one read.
//
// What follows the search (events), by features listed; in brackets with one CTA
// of the last feature doing the update, 256 samples after another:
//   15,000 samples       21: 43 us (178)   300: 51 (182)   5,050: 248 (412)
//   32,766 samples       21: 57 us (403)   300: 82 (414)   5,050: 602 (800)
//   600 samples          21: 29 us (35)    595: 42 (40)    5,050: 146 (153)
//   20x20 / 19,997       78,460: 5.3 ms (6.0), the whole round
__global__ void __launch_bounds__(kTailThreads + 32, 2) k_plateau(const __grid_constant__ JobDesc J) {
    RoundState *rs = J.rs;
    // (the same for every CTA: only the last cluster writes them, when all have read)
    const int32_t status = rs->status, count = rs->cand_count, r0 = rs->rounds;
    const float m = rs->screen_min;
    if (status != VJB_OK || count == 0) return;
    __shared__ TailShared<kPlateauCtas> S;
    __shared__ Candidate mine[kTailThreads / 32 + 1];
    __shared__ bool last;
    auto cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int64_t c0 = blockIdx.x; c0 < count; c0 += (int64_t)kTailCands * gridDim.x) {
        const int feats = (int)min((int64_t)kTailCands, (count - c0 + gridDim.x - 1) / gridDim.x);
        for (int i = warp; i < feats * 32; i += (int)blockDim.x >> 5) {
            const int32_t f = J.cand_ids[c0 + (i >> 5) * (int64_t)gridDim.x];
            const RunResult r = rescan_run(J.rows + (size_t)f * J.npad, J.npad / 32, i & 31, J.v, lane);
            if (lane == 0) S.runs[i] = r;
        }
        __syncthreads();
        if (warp < feats) {
            const int64_t c = c0 + warp * (int64_t)gridDim.x;
            const Candidate cd = combine_runs(J, J.cand_ids[c], S.runs[warp * 32 + lane], lane);
            if (lane == 0) J.cands[c] = cd;
        }
        __syncthreads();
    }
    if (lane == 0) __threadfence();
    cluster.sync();
    if (rank == 0 && warp == 0) {
        bool l = false;
        if (lane == 0) {
            __threadfence();
            l = atomicAdd(&rs->done_rescan, 1u) == gridDim.x / kPlateauCtas - 1;
            __threadfence();
        }
        l = __shfl_sync(0xffffffffu, (int)l, 0) != 0;
        if (lane < kPlateauCtas) *cluster.map_shared_rank(&last, lane) = l;
    }
    cluster.sync();
    if (!last) return;  // the whole cluster
    if (rank == 0 && tid == 0) rs->done_rescan = 0u;
    // the best of the list: a share a CTA, then of theirs
    Candidate b = no_candidate();
    for (int k = rank * (int)blockDim.x + tid; k < count; k += kPlateauCtas * (int)blockDim.x) {
        const Candidate c = load_candidate(J.cands + k);
        if (cand_less(c, b)) b = c;
    }
    auto warp_best = [](Candidate x) {
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            const Candidate o = cand_shfl_xor(x, d);
            if (cand_less(o, x)) x = o;
        }
        return x;
    };
    b = warp_best(b);
    if (lane == 0) mine[warp] = b;
    __syncthreads();
    if (warp == 0) {
        b = warp_best(lane < kTailThreads / 32 + 1 ? mine[lane] : no_candidate());
        if (lane < kPlateauCtas) cluster.map_shared_rank(&S, lane)->found[rank] = b;
    }
    cluster.sync();
    tail_update(J, S, best_found(S.found, kPlateauCtas), count, m, r0);
}

cudaError_t set_tail_limits() {
    return cudaFuncSetAttribute(k_tail, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// A launch of `clusters` clusters of CTAS.
template <int CTAS>
struct ClusterLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    ClusterLaunch(int clusters, cudaStream_t st) {
        cfg.gridDim = dim3(clusters * CTAS);
        cfg.blockDim = dim3(kTailThreads + 32);
        cfg.stream = st;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = CTAS;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
};

int plateau_clusters() {
    int n = 0;
    ClusterLaunch<kPlateauCtas> l(1, nullptr);
    return cudaOccupancyMaxActiveClusters(&n, k_plateau, &l.cfg) == cudaSuccess && n > 0 ? n : 1;
}

cudaError_t launch_tail(const JobDesc &J, const float *bmin, int nbmin, int clusters, cudaStream_t st) {
    ClusterLaunch<kTailCtas> tail(1, st);
    const cudaError_t e = cudaLaunchKernelEx(&tail.cfg, k_tail, J, bmin, nbmin);
    if (e != cudaSuccess) return e;
    ClusterLaunch<kPlateauCtas> plateau(clusters, st);
    return cudaLaunchKernelEx(&plateau.cfg, k_plateau, J);
}

}  // namespace vjb
