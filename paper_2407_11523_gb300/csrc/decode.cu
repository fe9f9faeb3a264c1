// Launch-shape selection and launch of the decode kernel (the kernel itself
// is in decode_kernel.cuh, instantiated per variant in decode_<variant>.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

#include "bpq_internal.h"
#include "decode_launch.h"

namespace bpq {

namespace {

int state_arrays(int variant) { return decode_state_arrays(variant); }

DecodeKernelFn pick(int variant, int npt, bool trace, int layout) {
    const bool split = layout != 0, full = layout == 2 && !trace;
    switch (variant) {
        case BPQ_PLAIN: return full ? pick_plain_full(npt) : pick_plain(npt, trace, split);
        case BPQ_MOMENTUM: return full ? pick_momentum_full(npt) : pick_momentum(npt, trace, split);
        case BPQ_ADAGRAD: return full ? pick_adagrad_full(npt) : pick_adagrad(npt, trace, split);
        case BPQ_EWAINIT: return full ? pick_ewainit_full(npt) : pick_ewainit(npt, trace, split);
        case BPQ_AEWA: return full ? pick_aewa_full(npt) : pick_aewa(npt, trace, split);
    }
    return nullptr;
}

DecodeKernelFn pick_pair(int variant, int mode, int layout) {
    const bool full = layout == 2;
    switch (variant) {
        case BPQ_PLAIN: return full ? pick_plain_pair_full(mode) : pick_plain_pair(mode);
        case BPQ_MOMENTUM: return full ? pick_momentum_pair_full(mode) : pick_momentum_pair(mode);
        case BPQ_ADAGRAD: return full ? pick_adagrad_pair_full(mode) : pick_adagrad_pair(mode);
        case BPQ_EWAINIT: return full ? pick_ewainit_pair_full(mode) : pick_ewainit_pair(mode);
    }
    return nullptr;
}

}  // namespace

bool decode_uses_pairs(const bpq_tanner *t, int variant, bool trace) {
    if (trace || !t->split || variant < BPQ_PLAIN || variant > BPQ_EWAINIT) return false;
    if (t->shots_per_thread == 1) return false;
    if (t->shots_per_thread == 2) return true;
    // automatic: where the stored launch shape fits two shots per thread
    LaunchShape s;
    const std::string keep = bpq_last_error();
    const bool fits = decode_pair_shape(t, variant, &s) == BPQ_OK;
    set_error(keep);
    return fits;
}

int decode_pair_shape(const bpq_tanner *t, int variant, LaunchShape *s) {
    const int nodes = t->N > t->M ? t->N : t->M;
    const int nstate = state_arrays(variant), n_pad = (t->N + 3) & ~3;
    const uint32_t slots = (uint32_t)(4 * n_pad + 4);  // float2 slots
    // per group: two vote words (16 bytes) | float2 slots | float2 state
    const size_t group_bytes = kPairVoteBytes + 8 * (size_t)slots + 8 * (size_t)(nstate * n_pad);
    const size_t one_smem = pair_offsets(variant, true, t->M, n_pad).groups + group_bytes;
    int T = t->threads_per_shot, gpc = t->shots_per_cta;
    if (T <= 0) {
        // Automatic.  Two nodes per thread, except that
        //  * a code of at most 96 nodes takes one warp per group (no barrier, warp
        //    votes only: planar d = 7, 10^6 shots, EWAInit 2.97 ms against 3.29 with
        //    two warps, d = 6 0.94 against 1.07; d = 8, four nodes per lane, 1.61
        //    against 1.49);
        //  * above 512 nodes 256 threads where shared memory holds two such CTAs
        //    (more nodes per thread but more shots per SM: plain BP on planar d =
        //    25, 30001 shots, 18.9 ms against 23.0, d = 21 11.9 against 13.7); with
        //    variant state, which leaves room for fewer shots, only up to three
        //    nodes for most threads (60000 shots, EWAInit at p = 0.08, two nodes /
        //    256 threads: d = 18 7.02 / 6.72, toric d = 18 6.57 / 5.82, d = 20 8.32 /
        //    8.36, planar d = 20 9.22 / 9.37; Momentum at p = 0.03, toric d = 20 5.76 /
        //    6.08);
        //  * above 1536 nodes three per thread, as the one CTA per SM has more than
        //    768 threads otherwise (planar d = 31, 20000 shots, p = 0.03, two / three
        //    nodes: Momentum 12.4 / 12.0, EWAInit 4.50 / 4.26, AdaGrad 16.0 / 15.3).
        // One group per CTA but for the one-warp groups (planar d = 11 with 128
        // threads: 4.41 against 4.56).
        T = (((nodes + 1) / 2 + 31) / 32) * 32;
        if (nodes <= 96) T = 32;
        else if (nodes > 512 && (nstate == 0 || nodes <= 672) && 2 * (one_smem + 1024) <= 228 * 1024) T = 256;
        else if (nodes > 1536) T = (((nodes + 2) / 3 + 31) / 32) * 32;
        if (gpc <= 0) gpc = T == 32 ? 8 : 1;
    } else if ((nodes + T - 1) / T > 2) {
        return fail(BPQ_EINVAL, "two shots per thread take at most two nodes per thread");
    }
    if (T % 32 || T < 32 || T > kMaxThreadsPerShot)
        return fail(BPQ_EINVAL, "threads per shot group must be a multiple of 32 in [32, 1024]");
    const int npt = (nodes + T - 1) / T;
    const int max_groups = T == 32 ? kMaxPairGroupsPerCta : 15;
    if (gpc <= 0) gpc = 256 / T > 0 ? 256 / T : 1;  // about 256 threads per CTA
    if (gpc > max_groups) gpc = max_groups;
    while (gpc > 1 && gpc * T > 1024) --gpc;
    s->T = T;
    s->G = T / 32;
    s->npt = npt;
    s->groups_per_cta = gpc;
    s->n_pad = n_pad;
    s->slots_floats = slots;
    s->group_bytes = (uint32_t)group_bytes;
    // The table of byte offsets for one group per CTA and for one-warp groups
    // (these have their size at compile time: planar d = 5, 10^6 shots, plain 4.68 ->
    // 4.34 ms; d = 7, 500000 shots, Momentum 5.82 -> 5.53, EWAInit 1.82 -> 1.75),
    // unless the 16-bit table, half its size, brings a third more CTAs onto an SM
    // (64 registers a thread: 1024 threads).  Byte offsets / 16 bits, 60000 shots,
    // p = 0.08, EWAInit, ms: planar d = 18 (2 / 3 CTAs of 256) 7.39 / 6.72, toric d =
    // 18 (2 / 3) 6.30 / 5.82, planar d = 22 (1 / 2 of 480) 16.1 / 13.4, toric d = 22
    // 13.6 / 11.0; d = 16 (3 / 4) 4.67 / 4.62; but with the same or nearly the same
    // number toric d = 15 3.31 / 3.48, planar d = 11 Momentum (7 / 8 of 128), 150000
    // shots, p = 0.03, 2.61 / 3.08.
    const size_t wide = one_smem + (size_t)(gpc - 1) * group_bytes;
    const size_t narrow = pair_offsets(variant, false, t->M, n_pad).groups + (size_t)gpc * group_bytes;
    auto resident = [&](size_t smem) {
        return std::min<size_t>(std::max(1, 1024 / (T * gpc)), 228 * 1024 / (smem + 1024));
    };
    const bool offsets = (gpc == 1 || T == 32) && wide <= 227 * 1024 && 3 * resident(narrow) < 4 * resident(wide);
    s->pair_mode = !offsets ? kPairGroups : gpc == 1 ? kPairOne : kPairWarps;
    s->smem = offsets ? wide : narrow;
    if (s->smem > 227 * 1024) return fail(BPQ_EINVAL, "shared memory of the launch shape exceeds 227 KB");
    return BPQ_OK;
}

namespace {
// Shape of the one-shot-per-thread kernels with T threads per shot and gpc
// shot groups per CTA (0: about 256 threads per CTA).
int one_shot_shape(const bpq_tanner *t, int variant, int T, int gpc, LaunchShape *s) {
    const int nodes = t->N > t->M ? t->N : t->M;
    if (T % 32 || T < 32 || T > kMaxThreadsPerShot)
        return fail(BPQ_EINVAL, "threads per shot must be a multiple of 32 in [32, 1024]");
    const int npt = (nodes + T - 1) / T;
    if (npt > kMaxNodesPerThread) return fail(BPQ_EINVAL, "too few threads per shot for this code");
    if (npt > 2 && T > 512) return fail(BPQ_EINVAL, "more than two nodes per thread needs at most 512 threads");
    // one-warp groups synchronise with __syncwarp; larger groups take one of
    // the 15 named barriers
    const int max_groups = T == 32 ? kMaxGroupsPerCta : 15;
    const int max_threads = npt <= 2 ? 1024 : 512;
    if (gpc <= 0) gpc = 256 / T > 0 ? 256 / T : 1;  // about 256 threads per CTA
    if (gpc > max_groups) gpc = max_groups;
    while (gpc > 1 && gpc * T > max_threads) --gpc;
    s->T = T;
    s->G = T / 32;
    s->npt = npt;
    s->groups_per_cta = gpc;
    s->n_pad = (t->N + 3) & ~3;
    // message slots (+ the zero slot, padded), state
    s->slots_floats = (uint32_t)(4 * s->n_pad + 4);
    const int nstate = state_arrays(variant < 0 ? BPQ_MOMENTUM : variant);
    s->group_bytes = (uint32_t)(4 * s->slots_floats + 4 * nstate * s->n_pad);
    s->smem = kSmemHeader + t->table.size() + (size_t)12 * s->n_pad + (size_t)gpc * s->group_bytes;
    if (s->smem > 227 * 1024) return fail(BPQ_EINVAL, "shared memory of the launch shape exceeds 227 KB");
    // the initial messages, unless they cost a resident CTA (48 registers a
    // thread: 1280 threads per SM).  Without and with them: AdaGrad on xzzx
    // d = 7, 5.7 iterations a shot, 200000 shots, 1.30 and 1.24 ms; AEWA on planar
    // d = 11, 11.3 iterations in a shot's last run, 10^5 shots, 11.3 and 11.2
    const size_t init = 16 * (size_t)s->n_pad, by_threads = std::max(1, 1280 / (T * gpc));
    auto resident = [&](size_t smem) { return std::min<size_t>(by_threads, 228 * 1024 / (smem + 1024)); };
    s->init_bytes = 0;
    if (s->smem + init <= 227 * 1024 && resident(s->smem + init) == resident(s->smem)) {
        s->init_bytes = (uint32_t)init;
        s->smem += init;
    }
    return BPQ_OK;
}
}  // namespace

int decode_launch_shape(const bpq_tanner *t, int variant, LaunchShape *s) {
    const int nodes = t->N > t->M ? t->N : t->M;
    const int T = t->threads_per_shot > 0 ? t->threads_per_shot : (((nodes + 1) / 2 + 31) / 32) * 32;
    return one_shot_shape(t, variant, T, t->shots_per_cta, s);  // automatic: two nodes per thread
}

namespace {
// Shape of a code in the batched kernel with npt (1 or 2) nodes per thread:
// the fewest threads per shot group that cover max(N, M), and as many shot
// groups as fit in kBatchThreads threads and 227 KB of shared memory.
int batch_shape_npt(const bpq_tanner *t, int variant, int npt, LaunchShape *s) {
    const int nodes = t->N > t->M ? t->N : t->M;
    const int T = (((nodes + npt - 1) / npt + 31) / 32) * 32;
    if (T > kBatchThreads) return fail(BPQ_EINVAL, "code too large for the batched kernel");
    const int max_groups = T == 32 ? kMaxGroupsPerCta : 15;
    int gpc = kBatchThreads / T;
    if (gpc > max_groups) gpc = max_groups;
    s->T = T;
    s->G = T / 32;
    s->npt = npt;
    s->n_pad = (t->N + 3) & ~3;
    s->slots_floats = (uint32_t)(4 * s->n_pad + 4);
    const int nstate = state_arrays(variant);
    s->group_bytes = (uint32_t)(4 * s->slots_floats + 4 * nstate * s->n_pad);
    const size_t fixed = kSmemHeader + kDescBytes + t->table.size() + (size_t)12 * s->n_pad;
    while (gpc > 1 && fixed + (size_t)gpc * s->group_bytes > 227 * 1024) --gpc;
    s->groups_per_cta = gpc;
    s->smem = fixed + (size_t)gpc * s->group_bytes;
    if (s->smem > 227 * 1024) return fail(BPQ_EINVAL, "a code of the batch needs more than 227 KB of shared memory");
    return BPQ_OK;
}
}  // namespace

int decode_batch_shape(const bpq_tanner *t, int variant, LaunchShape *s) {
    if (t->batch_nodes_per_thread > 0) return batch_shape_npt(t, variant, t->batch_nodes_per_thread, s);
    // automatic: the node count per thread that keeps the most node slots of
    // a CTA busy (groups x nodes / (npt x kBatchThreads)); on a tie two nodes
    // per thread, whose twice as many groups balance the item's shots better
    LaunchShape one, two;
    const std::string keep = bpq_last_error();
    const int rc1 = batch_shape_npt(t, variant, 1, &one);
    const int rc2 = batch_shape_npt(t, variant, 2, &two);
    if (rc2) {
        if (rc1) return rc2;
        *s = one;
    } else {
        *s = !rc1 && 2 * one.groups_per_cta > two.groups_per_cta ? one : two;
    }
    set_error(keep);
    return BPQ_OK;
}

namespace {

// Launch of a small batch (decode_small.cu): one CTA per shot, `lanes` lanes
// per node, every shot resident at once (or in two rounds).  Returns false if the batch, the code
// or the handle's launch preferences call for the queue kernels.
//
// Measured (kernel and launch, EWAInit or Momentum, us), against one node per
// thread in the queue kernel: planar d = 9, 150 shots: 4 lanes 66, queue 92;
// 300 shots: 4 lanes 107, 2 lanes 80, 1 lane 79, queue 91; 600: 2 lanes 103,
// 1 lane 92, queue 94; toric d = 15, 150 shots: 2 lanes 102, 1 lane 86, queue
// 95.  More lanes shorten a shot's chain but add instructions (every lane of a
// node computes its posterior), so they pay while an SM holds at most about
// 640 threads of them; one lane per node pays (no queue reset, no table
// staging) while every shot has a CTA of its own.
bool launch_small(const bpq_tanner *t, DecodeArgs &a, int variant, cudaStream_t st, int *rc) {
    if (a.split == 0 || t->threads_per_shot || t->shots_per_cta || t->shots_per_thread) return false;
    const int nodes = t->N > t->M ? t->N : t->M;
    const long shots_per_sm = ((long)a.B + t->num_sms - 1) / t->num_sms;
    int lanes = 4;
    while (lanes > 1 && lanes * nodes * shots_per_sm > 640) lanes /= 2;
    // AdaGrad on a large code fills the SM's issue slots with fewer threads (304
    // shots, us, this / one node per thread in the queue kernel: toric d = 15 (900
    // nodes of an SM) 162 / 124, planar d = 15 (842) 111 / 144)
    if (variant == BPQ_ADAGRAD && nodes > 256 && nodes * shots_per_sm > 864) return false;
    // Large codes, whose CTAs nearly fill an SM, take two rounds of them: 304 shots,
    // us, this / one node per thread in the queue kernel / two: Momentum at p = 0.05
    // planar d = 18 105 / 126 / 172, toric d = 20 134 / 158 / 195, planar d = 22 228 /
    // 261 / 236; EWAInit at p = 0.08 97 / 110 / 157, 127 / 133 / 178, 153 / 165 / 215.
    // So do the tiniest, whose CTAs are over first where the queue kernel starts its
    // CTAs and tables: 7000 shots of Momentum, this / queue: planar d = 2 62 / 85, d =
    // 3 42 / 60, d = 4 58 / 69
    const int rounds = nodes <= 32 || (nodes > 512 && variant != BPQ_ADAGRAD && variant != BPQ_AEWA) ? 2 : 1;
    if (nodes > 1024 || shots_per_sm > 32 * rounds) return false;
    const int threads = (lanes * nodes + 31) / 32 * 32;
    const size_t smem = 16 * (size_t)((t->N + 3) & ~3);
    SmallKernelFn fn = pick_small(variant, lanes);
    int per_sm = 0;
    if (!fn || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess ||
        shots_per_sm > rounds * per_sm)
        return false;
    if (t->debug_checks && !(fn = pick_debug_small(variant, lanes))) return false;
    a.n_pad = (t->N + 3) & ~3;
    const bool unclipped = a.split == 2 && variant != BPQ_ADAGRAD;
    if (t->debug_checks) {  // the checked copy does not reset the error word, which any CTA may set
        *rc = cuda_check(cudaMemsetAsync(a.work, 0, 8, st), "workspace reset");
        if (*rc) return true;
    }
    fn<<<(unsigned)a.B, threads, smem, st>>>(a, variant == BPQ_AEWA ? 11 : 1, unclipped ? INFINITY : a.clip2);
    *rc = cuda_check(cudaGetLastError(), "decode launch");
    return true;
}

// One node per thread instead of the automatic two for batches of fewer than three
// shots per resident two-node group: they are bound by their slowest shots, whose
// iterations are shorter then (kernel and launch, us, two nodes against one:
// planar d = 9 Momentum, p = 0.05, 1000 shots 139 / 112, 5000 (3.3 per group) 209 /
// 183; toric d = 15 Momentum 912 (1.2) 198 / 168, 1520 (2) 234 / 225, 2432 (3.2) 293 /
// 308; at p = 0.03 planar d = 18, 700 (1.2) plain 213 / 160, Momentum 220 / 158,
// planar d = 15 Momentum 1500 211 / 164; EWAInit toric d = 20 700 126 / 109).  Once
// an SM is full a shot of one node per thread costs it more, so where most shots run
// long two nodes are ahead on large codes: Momentum at p = 0.08 toric d = 15, 1500,
// 353 / 391, d = 20, 700 391 / 440, planar d = 18, 700 344 / 384; but the prior is
// not the host's to read.  Plain BP, most of whose shots run long at p = 0.03 too,
// takes two nodes above 700 (toric d = 20, 700 shots 186 / 215).
constexpr long one_node_half_shots(int variant, int nodes) {
    return variant == BPQ_PLAIN && nodes > 700 ? 0 : 6;
}

}  // namespace

// Every kernel that decode_launch can pick for this variant and table layout,
// whatever the batch and the stored shape.  The runtime loads a kernel when it is
// first asked about it (CUDA's lazy loading), so asking about all of them leaves
// no load, and no allocation for one, to a later call of another batch size.
int decode_preload(const bpq_tanner *t, int variant) {
    if (variant < BPQ_PLAIN || variant > BPQ_AEWA) return BPQ_OK;  // refused later
    const int layout = t->full ? 2 : t->split ? 1 : 0;
    static std::atomic<uint32_t> loaded[kMaxPreloadDevices];  // bit per (checked, layout, variant)
    const uint32_t bit = 1u << ((t->debug_checks ? 15 : 0) + 5 * layout + variant);
    std::atomic<uint32_t> *done = t->device < kMaxPreloadDevices ? &loaded[t->device] : nullptr;
    if (done && (done->load(std::memory_order_acquire) & bit)) return BPQ_OK;
    const bool pairs = layout && variant != BPQ_AEWA;
    std::vector<const void *> fns;
    auto add = [&](auto *fn) {
        if (fn) fns.push_back(reinterpret_cast<const void *>(fn));
    };
    for (int npt = 1; npt <= 3; ++npt)  // three and more: one kernel
        add(t->debug_checks ? pick_debug(variant, npt, false, 0, layout) : pick(variant, npt, false, layout));
    for (int mode = kPairGroups; pairs && mode <= kPairWarps; ++mode)
        add(t->debug_checks ? pick_debug(variant, 1, true, mode, layout) : pick_pair(variant, mode, layout));
    for (int lanes = 1; layout && lanes <= 4; lanes *= 2)
        add(t->debug_checks ? pick_debug_small(variant, lanes) : pick_small(variant, lanes));
    for (const void *fn : fns) {
        cudaFuncAttributes attr;
        const int rc = cuda_check(cudaFuncGetAttributes(&attr, fn), "kernel load");
        if (rc) return rc;
    }
    if (done) done->fetch_or(bit, std::memory_order_release);
    return BPQ_OK;
}

namespace {
// Threads of a kernel's launch shape that an SM holds at once.  Automatic pairs need
// more than half of the one-shot kernel's if they are one group, all of which waits
// at its barriers: planar d = 23, one CTA of 512 threads against two, 20000 shots at p
// = 0.03, one / two shots per thread: Momentum 4.01 / 4.97 ms, EWAInit 1.47 / 1.95; p
// = 0.08 12.5 / 15.2, 4.70 / 5.79.  Two groups are ahead with fewer: planar d = 25
// plain, two of 256 threads against two of 608, 30001 shots at p = 0.06 19.4 / 18.9.
int resident_threads(DecodeKernelFn fn, const LaunchShape &s) {
    int per_sm = 0;
    if (!fn || allow_smem(fn, kMaxDynamicSmem, "cudaFuncSetAttribute") != BPQ_OK ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, s.T * s.groups_per_cta, s.smem) != cudaSuccess)
        return 0;
    return per_sm * s.T * s.groups_per_cta;
}
constexpr long kInitShotsPerGroup = 4;

}  // namespace

int decode_launch(const bpq_tanner *t, DecodeArgs &a, int variant, bool trace, cudaStream_t st) {
    int small_rc = BPQ_OK;
    if (!trace && launch_small(t, a, variant, st, &small_rc)) return small_rc;
    LaunchShape s;
    bool pairs = decode_uses_pairs(t, variant, trace);
    if (pairs && t->shots_per_thread == 0) {
        // automatic choice: a pair's iteration does two shots' work, so a
        // batch's tail (its slowest shots) runs longer; pairing pays only
        // once each resident one-shot group would decode many shots.
        // Measured on GB300, one shot per thread against two (ms; shots per
        // resident one-shot group).  Plain and Momentum BP, whose shots mostly
        // run long, cross early: planar d = 13 Momentum 60000 (79), p = 0.08 and
        // 0.03, 8.94 / 8.38 and 1.92 / 1.95, toric d = 8 Momentum 200000 (66) 3.78 /
        // 3.60 and 0.95 / 1.03, planar d = 11 plain 100000 (82) 4.22 / 4.12, at p =
        // 0.03 150000 (123) 2.83 / 2.98, d = 25 plain 10000 (66) 6.00 / 5.97; one-warp
        // pair groups: planar d = 7 Momentum 500000 (205) 6.39 / 5.53.  EWAInit and
        // AdaGrad converge in few iterations, so that the slowest shots weigh more:
        // planar d = 11 EWAInit 100000 (82) 1.50 / 1.56, d = 13 100000 (110) 2.71 /
        // 2.73, d = 9 200000 (132) 1.75 / 1.77, 400000 (263) 3.43 / 3.38; d = 7 300000
        // (123) 0.957 / 1.011, 500000 (205) 1.85 / 1.75; large codes again earlier,
        // without padding above all: toric d = 15, 60000 (99), p = 0.08 3.45 / 3.31, p = 0.03
        // 1.21 / 1.24; planar d = 15, 60000 (79) 4.01 / 3.95 and 1.23 / 1.32; AdaGrad,
        // 60000, p = 0.08 and 0.03: toric d = 15 13.7 / 13.5 and 3.23 / 3.44, d = 13
        // 9.27 / 9.16 and 2.15 / 2.34, planar d = 15 17.4 / 16.8 and 3.91 / 4.05.  A
        // code whose one-shot group is one warp too gains nothing, 10^6 shots (205):
        // planar d = 4 plain 0.75 / 0.96, Momentum 1.57 / 1.83, d = 5 plain 1.58 /
        // 1.86, EWAInit 1.75 / 1.91, AdaGrad 2.25 / 2.66; but Momentum with two nodes
        // per lane at p = 0.08: d = 5 8.52 / 8.08, d = 6 10.8 / 10.2.
        LaunchShape one;
        int per_sm = 0;
        DecodeKernelFn f1 = nullptr;
        if (decode_launch_shape(t, variant, &one) == BPQ_OK && (f1 = pick(variant, one.npt, false, a.split)) &&
            allow_smem(f1, kMaxDynamicSmem, "cudaFuncSetAttribute") == BPQ_OK &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f1, one.T * one.groups_per_cta, one.smem) ==
                cudaSuccess &&
            decode_pair_shape(t, variant, &s) == BPQ_OK) {
            const int one_threads = per_sm * one.T * one.groups_per_cta;
            pairs = (long)a.B >= pair_shots_per_group(variant, s.T, one.T, std::max(t->N, t->M), t->full) *
                                     (long)per_sm * t->num_sms * one.groups_per_cta;
            if (pairs) {
                const int threads = resident_threads(pick_pair(variant, s.pair_mode, a.split), s);
                pairs = threads > s.T || 2 * threads > one_threads;
            }
        }
    }
    int rc = pairs ? decode_pair_shape(t, variant, &s) : decode_launch_shape(t, variant, &s);
    if (rc) return rc;
    DecodeKernelFn fn = nullptr;
    if (t->debug_checks) {
        fn = trace ? nullptr : pick_debug(variant, s.npt, pairs, s.pair_mode, a.split);
        if (!fn)
            return fail(BPQ_EINVAL, "no bounds-checked kernel for this launch (plain, Momentum, AdaGrad or EWAInit BP, "
                                    "at most two nodes per thread, not a trace)");
    } else {
        fn = pairs ? pick_pair(variant, s.pair_mode, a.split) : pick(variant, s.npt, trace, a.split);
    }
    if (!fn) return fail(BPQ_EINVAL, "no kernel for this variant (AEWA-BP has no trace mode)");
    rc = allow_smem(fn, kMaxDynamicSmem, "cudaFuncSetAttribute");
    if (rc) return rc;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, s.T * s.groups_per_cta, s.smem);
    if (e != cudaSuccess || per_sm < 1) return fail(BPQ_ECUDA, "launch shape does not fit on an SM");
    const int nodes = t->N > t->M ? t->N : t->M;
    const long groups = (long)per_sm * t->num_sms * s.groups_per_cta;
    if (!pairs && !trace && s.npt == 2 && !t->threads_per_shot && !t->shots_per_cta && nodes <= kMaxThreadsPerShot &&
        2L * a.B < one_node_half_shots(variant, nodes) * groups) {
        rc = one_shot_shape(t, variant, (nodes + 31) / 32 * 32, 0, &s);
        if (rc) return rc;
        fn = t->debug_checks ? pick_debug(variant, s.npt, false, 0, a.split) : pick(variant, s.npt, false, a.split);
        if (!fn) return fail(BPQ_EINVAL, "no kernel for this variant");
        rc = allow_smem(fn, kMaxDynamicSmem, "cudaFuncSetAttribute");
        if (rc) return rc;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, s.T * s.groups_per_cta, s.smem);
        if (e != cudaSuccess || per_sm < 1) return fail(BPQ_ECUDA, "launch shape does not fit on an SM");
    }
    // The initial messages' table, made by every CTA, pays from some shots per group
    // on (kernel and launch, us, with / without it, p = 0.03): toric d = 20 EWAInit,
    // 1500 shots (3.3 per group) 151 / 145; d = 3, 8000 (1.3) 26.3 / 25.4; planar d = 2
    // plain, 8000, p = 0.08 92.5 / 87.8; planar d = 5 Momentum, 20000 (4.1) 132 / 146, d =
    // 13 EWAInit, 4800 (5.2) 145 / 151.
    if (!pairs && !trace && (long)a.B < kInitShotsPerGroup * per_sm * t->num_sms * s.groups_per_cta) {
        s.smem -= s.init_bytes;
        s.init_bytes = 0;
    }
    const int threads = s.T * s.groups_per_cta;
    long ctas = (long)per_sm * t->num_sms;
    const long per_cta = (long)s.groups_per_cta * (pairs ? 2 : 1);
    const long need = (a.B + per_cta - 1) / per_cta;
    if (ctas > need) ctas = need;
    if (ctas < 1) ctas = 1;
    a.G = s.G;
    a.n_pad = s.n_pad;
    a.slots_floats = s.slots_floats;
    a.group_bytes = s.group_bytes;
    a.init_bytes = pairs ? 0 : s.init_bytes;
    rc = cuda_check(cudaMemsetAsync(a.work, 0, 8, st), "workspace reset");  // the shot queue, the error word
    if (rc) return rc;
    fn<<<(unsigned)ctas, threads, s.smem, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(BPQ_ECUDA, std::string("decode launch: ") + cudaGetErrorString(e));
    return BPQ_OK;
}

}  // namespace bpq
