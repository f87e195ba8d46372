// Weight kernels of a boosting round (Sec. 2.3); the plain rounds' updates are
// part of their tail kernel (k_tail.cu), which shares k_update.cuh with these:
//  * k_init_weights: the initial weights of Table 2 (1/(2l) per face, 1/(2m)
//    per non-face) or caller-given weights, normalised (step 1).  One cluster.
//  * k_update_a (host-given stumps; k_bupdate in batches): the round's stump
//    applied to every sample: e_i (misclassified
//    or not) and FP64 partial sums of the misclassified and of all weight.
//    The last CTA to finish forms the error (step 2, exact given the FP32
//    weights), the threshold, beta and alpha (step 3), records the stump, and
//    derives the two factors of the update and renormalisation:
//        w_i <- w_i beta^(1 - e_i) / Z,   Z = M + beta (T - M),
//    M the misclassified weight and T the total (steps 4 and 1).
//  * k_update_b: applies those factors in FP64 and stores the FP32 weights in
//    both copies of the weight array; its last CTA forms the class totals of
//    the stored weights for the next search.
// FP64 is used only for the sums, the error, beta, alpha and the one multiply
// per sample of the renormalisation.
#include <cooperative_groups.h>
#include <math.h>

#include "k_update.cuh"

namespace vjb {

// k_init_weights: 1,024 threads as a cluster of 8 CTAs on 8 SMs.  GB300's FP64
// unit runs at a couple of lanes per clock per SM: one CTA of 1,024 threads
// took 64 us for 1,000 samples (every warp of it added the 32 warps' sums, one
// after another, five times) and 100 us for 15,000 (its own share of the FP64
// work); this form takes 15 us at 15,000 (ncu), and
// vjb_set_weights 107 -> 46 us there and 57 -> 26 us at 600.
constexpr int kInitCtas = 8, kInitThreads = 128, kInitWarps = kInitThreads / 32;

// Sum of one double per thread over the cluster in a fixed order: lanes by a
// butterfly, then the 32 warps' sums one after another.  `part` is this sum's
// place in every CTA's shared memory, `total` where this CTA's threads find the
// result; `adder` is the warp that adds up.
__device__ __forceinline__ void cluster_partial(double x, double *part) {
    x = warp_sum_d(x);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
}
__device__ __forceinline__ void cluster_total(double *part, double *all, double *total, int adder) {
    if ((int)threadIdx.x >> 5 != adder) return;
    const int lane = threadIdx.x & 31;
    auto cluster = cooperative_groups::this_cluster();
    static_assert(kInitCtas * kInitWarps == 32, "a lane per warp of the cluster");
    all[lane] = cluster.map_shared_rank(part, lane / kInitWarps)[lane % kInitWarps];
    __syncwarp();
    if (lane == 0) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 32; ++k) s += all[k];
        *total = s;
    }
}

__global__ void __cluster_dims__(kInitCtas, 1, 1) __launch_bounds__(kInitThreads)
    k_init_weights(const uint8_t *__restrict__ y, WeightLayout L, const float *__restrict__ w_in, double wf, double wn,
                   float *__restrict__ w, float *__restrict__ v, RoundState *rs) {
    __shared__ double part[3][kInitWarps], all[2][32], total[3];
    auto cluster = cooperative_groups::this_cluster();
    const int n = L.n, step = kInitCtas * kInitThreads, i0 = (int)(blockIdx.x * kInitThreads + threadIdx.x);
    // caller-given weights, or Table 2's: wf = 1/(2l) for faces, wn = 1/(2m) for non-faces
    double tot = 0.0;
    for (int i = i0; i < n; i += step) tot += w_in ? (double)w_in[i] : (y[i] ? wf : wn);
    cluster_partial(tot, part[0]);
    cluster.sync();
    cluster_total(part[0], all[0], &total[0], 0);
    if (threadIdx.x == 0) total[1] = 1.0 / total[0];
    __syncthreads();
    tot = total[0];
    const double r = total[1];
    double tp = 0.0, tn = 0.0;
    for (int i = i0; i < n; i += step) {
        const double wi = w_in ? (double)w_in[i] : (y[i] ? wf : wn);
        const float f = __double2float_rn(wi * r);
        w[i] = f;
        store_v(v, L, i, y[i] ? f : -f);
        if (y[i]) tp += (double)f; else tn += (double)f;
    }
    cluster_partial(tp, part[1]);
    cluster_partial(tn, part[2]);
    cluster.sync();
    if (blockIdx.x == 0) {
        cluster_total(part[1], all[0], &total[1], 0);
        cluster_total(part[2], all[1], &total[2], 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            tp = total[1];
            tn = total[2];
            v[n] = 0.f;
            rs->t_pos = tp;
            rs->t_neg = tn;
            rs->weight_sum = tp + tn;
            rs->status = VJB_OK;
            rs->cand_count = 0;
            rs->forced = 0;
            rs->done_rescan = rs->done_update_a = rs->done_update_b = 0u;
            rs->screen_min_bits = 0x7f800000u;
            rs->in_round = 0;
            if (!(tot > 0.0) || !isfinite(tot)) rs->flags |= kFlagBadWeights;
        }
    }
    cluster.sync();  // no CTA leaves while another reads its shared memory
}

cudaError_t launch_init_weights(const uint8_t *y, int faces, const WeightLayout &L, const float *w_in,
                                float *w, float *v, RoundState *rs, cudaStream_t st) {
    const double wf = 1.0 / (2.0 * faces), wn = 1.0 / (2.0 * (L.n - faces));
    k_init_weights<<<kInitCtas, kInitThreads, 0, st>>>(y, L, w_in, wf, wn, w, v, rs);
    return cudaGetLastError();
}

int update_grid(int n) {
    const int g = (n + kUpdateThreads - 1) / kUpdateThreads;
    return g < 1 ? 1 : (g > kUpdateMaxCtas ? kUpdateMaxCtas : g);
}

__global__ void __launch_bounds__(kUpdateThreads) k_update_a(const JobDesc J) {
    if (!update_a_block(J, blockIdx.x, false)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) store_threshold(J);
    if (!last_block_done(&J.rs->done_update_a, gridDim.x)) return;
    finish_a(J, gridDim.x);
}

__global__ void __launch_bounds__(kUpdateThreads) k_update_b(const JobDesc J) {
    if (!update_b_block(J, blockIdx.x, false)) return;
    if (!last_block_done(&J.rs->done_update_b, gridDim.x)) return;
    finish_b(J, gridDim.x);
}

cudaError_t launch_update_a(const JobDesc &J, cudaStream_t st) {
    k_update_a<<<update_grid(J.lay.n), kUpdateThreads, 0, st>>>(J);
    return cudaGetLastError();
}

cudaError_t launch_update_b(const JobDesc &J, cudaStream_t st) {
    k_update_b<<<update_grid(J.lay.n), kUpdateThreads, 0, st>>>(J);
    return cudaGetLastError();
}

// Batched: the blocks of all jobs in the round, flattened (job j owns blocks
// [ublock_base_j, ublock_base_j + update_grid(n_j))), each job's last block
// finishing it.  The same blocks and the same order of partial sums as the
// plain kernels, so a job's results do not depend on its batch.
template <bool A>
__global__ void __launch_bounds__(kUpdateThreads) k_bupdate(const JobDesc *__restrict__ jobs, BatchMeta *meta) {
    __shared__ int base[kMaxBatchJobs + 1];
    const int nj = meta->njobs;
    for (int j = threadIdx.x; j < nj; j += blockDim.x) base[j] = jobs[j].ublock_base;
    if (threadIdx.x == 0) base[nj] = meta->total_ublocks;
    __syncthreads();
    const int total = base[nj];
    for (int g = blockIdx.x; g < total; g += gridDim.x) {
        int lo = 0, hi = nj - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (base[mid] <= g) lo = mid;
            else hi = mid - 1;
        }
        const JobDesc &J = jobs[lo];
        const int blk = g - base[lo], nblocks = base[lo + 1] - base[lo];
        if (A) {
            if (!update_a_block(J, blk, true)) continue;
            if (blk == 0 && threadIdx.x == 0) store_threshold(J);
        } else {
            if (!update_b_block(J, blk, true)) continue;
        }
        if (last_block_done(A ? &J.rs->done_update_a : &J.rs->done_update_b, nblocks)) {
            if (A) finish_a(J, nblocks);
            else finish_b(J, nblocks);
        }
        __syncthreads();
    }
}

cudaError_t launch_bupdate_a(const JobDesc *jobs, BatchMeta *meta, int grid, cudaStream_t st) {
    k_bupdate<true><<<grid, kUpdateThreads, 0, st>>>(jobs, meta);
    return cudaGetLastError();
}

// End of a batched round: its outcome for the host.
__global__ void k_bend(const JobDesc *__restrict__ jobs, const BatchMeta *__restrict__ meta, BatchSeen *seen) {
    const int j = threadIdx.x;
    if (j == 0) seen->flags = meta->flags;
    if (j < meta->njobs) {
        const RoundState *rs = jobs[j].rs;
        seen->job[j] = JobSeen{rs->status, rs->rounds, rs->flags, 0};
    }
}

cudaError_t launch_bend(const JobDesc *jobs, const BatchMeta *meta, BatchSeen *seen, cudaStream_t st) {
    k_bend<<<1, kMaxBatchJobs, 0, st>>>(jobs, meta, seen);
    return cudaGetLastError();
}

cudaError_t launch_bupdate_b(const JobDesc *jobs, BatchMeta *meta, int grid, cudaStream_t st) {
    k_bupdate<false><<<grid, kUpdateThreads, 0, st>>>(jobs, meta);
    return cudaGetLastError();
}

}  // namespace vjb
