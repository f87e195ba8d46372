// Device pieces of the weight updates shared by the plain round's tail
// (k_tail.cu), the updates with a host-given stump and the batched ones
// (k_update.cu).
#pragma once

#include <math.h>

#include "vjb_device.cuh"
#include "vjb_haar.cuh"
#include "vjb_internal.cuh"

namespace vjb {

// The sample at position k of feature f's value order.
__device__ __forceinline__ int sample_at(const JobDesc &J, int32_t f, int k) {
    const int P = phys_of(k, J.npad / 32);
    return word_to_sample(entry_word(J.rows[(size_t)f * J.npad + P], P), J.lay);
}

__device__ __forceinline__ void store_v(float *v, const WeightLayout &L, int i, float x) {
    v[i] = x;
    if (L.dual && i < L.nb) v[L.off_b + rot_b(i)] = x;
}

// A stump's record (Sec. 2.3 step 3): beta = eps / (1 - eps), alpha = log(1 / beta).
__device__ __forceinline__ vjb_stump stump_record(int32_t f, int32_t p, int32_t theta, int32_t split, double eps) {
    vjb_stump st;
    st.feature = f;
    st.threshold = theta;
    st.polarity = p;
    st.split = split;
    st.error = eps;
    if (eps == 0.0) {
        st.beta = 0.0;
        st.alpha = INFINITY;
    } else {
        st.beta = eps / (1.0 - eps);
        st.alpha = log((1.0 - eps) / eps);
    }
    return st;
}

// Per-CTA reduction of three doubles into partials[3 * blk + k].  FP64 runs
// at a couple of lanes per clock per SM on this GPU, so a warp-wide FP64 add
// takes the FP64 pipe of its scheduler for tens of cycles: each value is
// summed by a warp of its own (warps 0, 1, 2 sit on different schedulers),
// lane l adding the threads l, l + 32, ... in order and the lanes then by a
// butterfly, 13 warp-wide adds a value instead of 40 spread over the CTA.
// The third value is reduced only where it can be non-zero (`third`, uniform
// over the launch), and its slot is 0 otherwise.
__device__ __forceinline__ void cta_partials(double a, double b, double c, bool third, double *partials, int blk) {
    __shared__ double red[3][kUpdateThreads];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    red[0][threadIdx.x] = a;
    red[1][threadIdx.x] = b;
    if (third) red[2][threadIdx.x] = c;
    __syncthreads();
    if (wp < 3) {
        double x = 0.0;
        if (wp < 2 || third) {
#pragma unroll
            for (int k = 0; k < kUpdateThreads / 32; ++k) x += red[wp][lane + 32 * k];
            x = warp_sum_d(x);
        }
        if (lane == 0) partials[3 * blk + wp] = x;
    }
}

// True in the CTA that finishes the last of `nblocks` blocks counted on
// `counter` (thread 0 decides, all threads learn).
__device__ __forceinline__ bool last_block_done(uint32_t *counter, int nblocks) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(counter, 1u) == (uint32_t)nblocks - 1;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Step 3-4, part 1, for the 256 samples (or sorted positions) of block `blk`:
// e_i and the block's FP64 sums of misclassified weight, of all weight and (for
// a host-given stump) of samples below the threshold.  The round state's
// fields are read in one trip with the status; false (nothing done, uniform
// over the CTA) when the job has stopped or, in a batch, sits this round out.
static __device__ bool update_a_block(const JobDesc &J, int blk, bool batched) {
    const int n = J.lay.n;
    const RoundState *rs = J.rs;
    const int32_t status = rs->status, in_round = rs->in_round, forced_i = rs->forced;
    const int32_t ff = rs->forced_feature, wf = rs->win_feature;
    const int32_t fp = rs->forced_polarity, wp = rs->win_polarity, ws = rs->win_split;
    const int32_t theta_f = rs->forced_threshold;
    if (status != VJB_OK || (batched && !in_round)) return false;
    const bool forced = forced_i != 0;
    const int32_t f = forced ? ff : wf;
    const int32_t p = forced ? fp : wp;
    const int32_t s = forced ? 0 : ws;
    const int k = blk * kUpdateThreads + threadIdx.x;
    double mw = 0.0, tw = 0.0, below = 0.0;
    if (k < n) {
        int i;
        bool h;
        if (!forced) {
            // sorted position k: the first s positions are "below" the threshold
            i = sample_at(J, f, k);
            const bool bl = k < s;
            h = (p > 0) ? bl : !bl;
        } else {
            i = k;
            const DevFeature d = J.feat[f];
            const int32_t val = haar_value(J.ii, J.ii_stride, J.win_w, d.type, d.x, d.y, d.w, d.h, i);
            h = (p > 0) ? (val < theta_f) : (val > theta_f);
            below = (p > 0) ? (val < theta_f) : (val <= theta_f);
        }
        const bool m = h != (J.y[i] != 0);
        J.miss[i] = m;
        const double wi = (double)J.w[i];
        tw = wi;
        if (m) mw = wi;
    }
    cta_partials(mw, tw, below, forced, J.partials, blk);
    return true;
}

// Sums of the three per-block partials over `nblocks` blocks by the finishing
// CTA in a fixed order, each value by a warp of its own (lane l adds blocks
// l, l + 32, ... in order, then the lanes by a butterfly); every thread gets
// them.  The third only where it can be non-zero (`third`), as in
// cta_partials.
__device__ __forceinline__ void sum_partials(const double *partials, int nblocks, bool third, double &a,
                                             double &b, double &c) {
    __shared__ double tot[3];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    if (wp < 3) {
        double x = 0.0;
        if (wp < 2 || third) {
            for (int k = lane; k < nblocks; k += 32) x += ((volatile const double *)partials)[3 * k + wp];
            x = warp_sum_d(x);
        }
        if (lane == 0) tot[wp] = x;
    }
    __syncthreads();
    a = tot[0];
    b = tot[1];
    c = tot[2];
}

// The searched stump's canonical threshold: p=+1 -> value at position s
// (max+1 at s = n); p=-1 -> value at position s-1 (min-1 at s = 0).
static __device__ int32_t stump_threshold(const JobDesc &J, int32_t f, int32_t p, int32_t s) {
    const int n = J.lay.n;
    const DevFeature d = J.feat[f];
    const uint16_t *row = J.rows + (size_t)f * J.npad;
    auto val_at = [&](int pos) {
        const int P = phys_of(pos, J.npad / 32);
        const int i = word_to_sample(entry_word(row[P], P), J.lay);
        return haar_value(J.ii, J.ii_stride, J.win_w, d.type, d.x, d.y, d.w, d.h, i);
    };
    if (p > 0) return (s < n) ? val_at(s) : val_at(n - 1) + 1;
    return (s > 0) ? val_at(s - 1) : val_at(0) - 1;
}

// One thread of the update's first block stores it in the round state before
// that block is counted, off the finishing block's path.
static __device__ void store_threshold(const JobDesc &J) {
    RoundState *rs = J.rs;
    if (!rs->forced) rs->win_theta = stump_threshold(J, rs->win_feature, rs->win_polarity, rs->win_split);
}

// Step 3-4, part 1, finish (after every block; the CTA's threads have summed
// the partials): the stump's FP64 error, threshold, beta and alpha, its
// record, and the update factors.  Three warps share the scalar work, so that
// the factors update b waits for do not queue behind the logarithm, the
// divisions of the diagnostics and their memory traffic (one thread did all of
// it in 7.5 us of a 13.3 us update at 24x24 / 15k): warp 0 the factors and
// the round state, warp 1 alpha and the stump record, warp 2 the diagnostics.
// Each value is computed exactly as one thread would.
static __device__ void update_a_finish(const JobDesc &J, double M, double T, double B) {
    RoundState *rs = J.rs;
    // the round state the parts read, taken before any part writes it
    const bool forced = rs->forced != 0;
    const int32_t f = forced ? rs->forced_feature : rs->win_feature;
    const int32_t p = forced ? rs->forced_polarity : rs->win_polarity;
    const int32_t s = forced ? 0 : rs->win_split;
    const int32_t r0 = rs->rounds;
    const int32_t cands = rs->cand_count;
    __syncthreads();
    const double eps = M / T;
    if (threadIdx.x == 0) {
        rs->last_cands = cands;
        rs->cand_count = 0;
        rs->forced = 0;
        rs->done_update_a = 0u;
        if (eps == 0.0) {
            // perfect stump: kept with alpha = +inf, training is over
            rs->rounds = r0 + 1;
            rs->status = VJB_DONE_PERFECT;
        } else if (eps >= 0.5) {
            // no stump does better than chance: not kept, training is over
            rs->status = VJB_DONE_NOGAIN;
        } else {
            const double beta = eps / (1.0 - eps);
            rs->rounds = r0 + 1;
            const double Z = M + beta * (T - M);
            rs->scale_hit = beta / Z;
            rs->scale_miss = 1.0 / Z;
        }
    } else if (threadIdx.x == 32) {
        int32_t theta, split = s;
        if (forced) {
            theta = rs->forced_threshold;
            split = (int32_t)B;
        } else {
            // written by another CTA in this launch: read past this SM's L1
            theta = *reinterpret_cast<volatile int32_t *>(&rs->win_theta);
        }
        const vjb_stump st = stump_record(f, p, theta, split, eps);
        *J.last = st;
        if (eps < 0.5 && r0 < J.stump_cap) J.stumps[r0] = st;
    } else if (threadIdx.x == 64) {
        // what the search saw of this stump, next to its FP64 error; the search
        // works in units of the current weight total T, so divide by it
        vjb_round_diag dg;
        dg.search_error = forced ? eps : ((double)rs->win_err_hi + (double)rs->win_err_lo) / T;
        dg.screen_error = forced ? (float)eps : (float)((double)J.ferr[f] / T);
        dg.screen_min = forced ? (float)eps : (float)((double)rs->screen_min / T);
        dg.candidates = forced ? 0 : cands;
        dg.forced = forced ? 1 : 0;
        if (r0 < J.stump_cap) J.diag[r0] = dg;
    }
}

// Step 4 and step 1 of the next round for the 256 samples of block `blk`.  The
// samples' miss flags, weights and labels are read in the same trip as the
// round state; false as for update_a_block.
static __device__ bool update_b_block(const JobDesc &J, int blk, bool batched) {
    const int i = blk * kUpdateThreads + threadIdx.x;
    const bool in = i < J.lay.n;
    const bool miss = in && J.miss[i];
    const float w0 = in ? J.w[i] : 0.f;
    const bool face = in && J.y[i] != 0;
    const RoundState *rs = J.rs;
    const int32_t status = rs->status, in_round = rs->in_round;
    const double scale_miss = rs->scale_miss, scale_hit = rs->scale_hit;
    if (status != VJB_OK || (batched && !in_round)) return false;
    double tp = 0.0, tn = 0.0;
    if (in) {
        const double scale = miss ? scale_miss : scale_hit;
        const float fw = __double2float_rn((double)w0 * scale);
        J.w[i] = fw;
        store_v(J.v, J.lay, i, face ? fw : -fw);
        if (face) tp = (double)fw; else tn = (double)fw;
    }
    cta_partials(tp, tn, 0.0, false, J.partials, blk);
    return true;
}

static __device__ void update_b_finish(const JobDesc &J, double P, double Q) {
    RoundState *rs = J.rs;
    rs->t_pos = P;
    rs->t_neg = Q;
    rs->weight_sum = P + Q;
    rs->done_update_b = 0u;
}

// The finishing CTA of update a / update b (all its threads).
static __device__ void finish_a(const JobDesc &J, int nblocks) {
    double M, T, B;
    // (the count below the threshold only for a host-given stump; read before
    // any part of the finish resets `forced`)
    sum_partials(J.partials, nblocks, J.rs->forced != 0, M, T, B);
    update_a_finish(J, M, T, B);
}

static __device__ void finish_b(const JobDesc &J, int nblocks) {
    double P, Q, unused;
    sum_partials(J.partials, nblocks, false, P, Q, unused);
    if (threadIdx.x == 0) update_b_finish(J, P, Q);
}

}  // namespace vjb
